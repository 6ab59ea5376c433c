"""The coarsest multigrid level as a matrix, solved in one launch.  A Q1 mesh of an odd number of
elements (or 2^3) is a hierarchy of one level, so the multigrid preconditioner is that solve alone:
to 1e-6 in FP64 and 1e-4 in FP32, so the flexible CG around it needs 2 and 3 iterations for 1e-10
when the matrix is the operator (one more allowed for the inner tolerance being tested every ten
iterations only, and for FP32's rounding)."""
import numpy as np
import pytest

import nhmf_inputs as inp
from tests.gpu_util import cuda, lib_or_fail

pytestmark = pytest.mark.gpu


# one block up to 4^3 nodes, clusters of 4, 8 and 16 blocks, rows in shared memory and in L2 (from
# 11^3 in FP64, 15^3 in FP32), 17^3 on the operator itself
@pytest.mark.parametrize("N", [2, 3, 5, 7, 9, 11, 13, 15, 17])
@pytest.mark.parametrize("bc,model,inclusions", [(1, 0, False), (2, 0, True), (2, 1, True)])
def test_coarse_solve_is_the_operators(N, bc, model, inclusions):
    import torch
    nhmf = lib_or_fail()
    w = inp.Workload("coarse", N, 1, 1.0, 1.5, bc, "scaled", 0.01, "normal", 1.0, 5100 + N, 5200 + N)
    prob = nhmf.Problem(N, 1, 1.0, 1.5, bc, model=model)
    if inclusions:
        nhmf.nhmf_set_material_factors(prob.ctx, cuda(inp.inclusion_factors(N)))
    prob.set_linearization(cuda(inp.draw_u(w)), 0 if model else nhmf.NHMF_CACHE_FP64 | nhmf.NHMF_CACHE_FP32)
    strat = nhmf.NHMF_ON_THE_FLY if model else nhmf.NHMF_CACHED
    b = cuda(inp.draw_du(w))
    x = torch.empty_like(b)
    for solver, most in ((nhmf.NHMF_SOLVER_GMG, 3), (nhmf.NHMF_SOLVER_MIXED_GMG, 4)):
        it, inner, rel = prob.linear_solve(b, x, solver=solver, strategy=strat, linear_rtol=1e-10)
        assert rel <= 1.01e-10 and it <= most and inner >= it, (solver, it, inner, rel)
    # a zero right-hand side, and one that is not finite
    it, inner, rel = prob.linear_solve(torch.zeros_like(b), x, solver=nhmf.NHMF_SOLVER_GMG, strategy=strat)
    assert it == 0 and float(x.abs().max()) == 0.0
    b[5] = float("nan")
    with pytest.raises(nhmf.NhmfError):
        prob.linear_solve(b, x, solver=nhmf.NHMF_SOLVER_GMG, strategy=strat)
    prob.close()
