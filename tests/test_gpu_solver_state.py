"""Solves on one context whose operator changes in between: the iterations that the solver replays
belong to the present material factors and caches (the true residual, by an apply outside the
replayed iterations, meets the tolerance)."""
import numpy as np
import pytest

import nhmf_inputs as inp
from tests.gpu_util import cuda, lib_or_fail

pytestmark = pytest.mark.gpu
RTOL = 1e-8


def workload(p, N):
    return inp.Workload("state", N, p, 1.0, 1.5, 1, "scaled", 0.01, "normal", 1.0, 4500 + N, 4600 + N)


@pytest.mark.parametrize("solver", ["NHMF_SOLVER_JACOBI_CG", "NHMF_SOLVER_MIXED_FCG"])
@pytest.mark.parametrize("p,N", [(1, 9), (2, 5)])
def test_material_factors_between_solves(solver, p, N):
    import torch
    nhmf = lib_or_fail()
    w = workload(p, N)
    prob = nhmf.Problem.from_workload(w)
    u, b = cuda(inp.draw_u(w)), cuda(inp.draw_du(w))
    prob.set_linearization(u, nhmf.NHMF_CACHE_FP64 | nhmf.NHMF_CACHE_FP32)
    x = torch.empty_like(b)
    fac = cuda(inp.inclusion_factors(N))
    for factors in (None, fac, 4.0 * fac, None, fac):
        nhmf.nhmf_set_material_factors(prob.ctx, factors)
        hold = torch.full((N ** 3,), np.nan, dtype=torch.float64, device="cuda:0")  # whatever was freed is reused
        for _ in range(2):
            _, _, rel = prob.linear_solve(b, x, solver=getattr(nhmf, solver), linear_rtol=RTOL)
            # the recursive residual that the solver tests drifts from the true one by rounding only
            assert rel <= 1.01 * RTOL, (factors is None, rel)
        del hold
    prob.close()


def test_spatial_cache_rebuilt_between_solves():
    import torch
    nhmf = lib_or_fail()
    w = workload(2, 5)
    prob = nhmf.Problem.from_workload(w)
    u, b = cuda(inp.draw_u(w)), cuda(inp.draw_du(w))
    x = torch.empty_like(b)
    other = []
    for k in range(4):
        prob.set_linearization(u * (1.0 - 0.2 * k), nhmf.NHMF_CACHE_SPATIAL)
        _, _, rel = prob.linear_solve(b, x, solver=nhmf.NHMF_SOLVER_JACOBI_CG, strategy=nhmf.NHMF_SPATIAL, linear_rtol=RTOL)
        assert rel <= 1.01 * RTOL, (k, rel)
        prob.set_linearization(u, 0)   # gives the cache back; the next one may lie elsewhere
        other.append(nhmf.Problem(5, 2, 1.0, 1.5, 1))
        other[-1].set_linearization(u, nhmf.NHMF_CACHE_SPATIAL)
    prob.close()
