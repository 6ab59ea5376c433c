"""The coarse solve's sums keep FP64's range and bits when its vectors are FP32: a material stiffer or
softer by 2^k changes the solution by 2^-k and nothing else.  The squares that the sums add lie
near 2^-k times the squares of the coarse residual (about 2^-14 to 2^-40 of a unit right-hand side),
so that at k = 112 they leave FP32's range while the vectors stay inside it."""
import numpy as np
import pytest

import nhmf_inputs as inp
from tests.gpu_util import cuda, lib_or_fail

pytestmark = pytest.mark.gpu
RTOL = 1e-9


@pytest.mark.parametrize("p,N", [(1, 8), (1, 6), (2, 6), (1, 9)])
@pytest.mark.parametrize("k", [112, 60, -60, -112])
@pytest.mark.parametrize("by", ["factors", "mu"])
def test_scaled_materials(p, N, k, by):
    import torch
    nhmf = lib_or_fail()
    w = inp.Workload("range", N, p, 1.0, 1.5, 1, "scaled", 0.01, "normal", 1.0, 4900 + N, 5000 + N)
    u, b = cuda(inp.draw_u(w)), cuda(inp.draw_du(w))
    b[torch.from_numpy(inp.dirichlet_mask(N, p, 1).reshape(-1)).cuda()] = 0.0  # identity rows do not scale
    got = []
    for e in (0, k):
        s = 2.0 ** e
        prob = nhmf.Problem(N, p, s, 1.5 * s, 1) if by == "mu" else nhmf.Problem(N, p, 1.0, 1.5, 1)
        if by == "factors":
            nhmf.nhmf_set_material_factors(prob.ctx, torch.full((N ** 3,), s, dtype=torch.float64, device="cuda:0"))
        prob.set_linearization(u, nhmf.NHMF_CACHE_FP64 | nhmf.NHMF_CACHE_FP32)
        x = torch.empty_like(b)
        it, inner, rel = prob.linear_solve(b, x, solver=nhmf.NHMF_SOLVER_MIXED_GMG, linear_rtol=RTOL)
        assert rel <= 1.01 * RTOL, (e, it, rel)
        got.append((it, inner, x * s))
        prob.close()
    (it0, inner0, x0), (it1, inner1, x1) = got
    # at k = 112 FP32 entries below 2^-14 of the largest are subnormal: absolute roundings 2^-37 of the
    # largest, below those of its own 24 bits
    assert abs(it1 - it0) <= 1 and abs(inner1 - inner0) <= 0.2 * inner0 + 10, (it0, it1, inner0, inner1)
    # two solutions with residuals of RTOL, condition number below 1e4
    assert float((x1 - x0).norm()) <= 2e4 * RTOL * float(x0.norm())
