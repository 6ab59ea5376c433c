"""The point code at very large volume ratios: an element stretched by F = diag(1 + a, 1 + b, 1), J =
(1 + a)(1 + b) up to the end of the FP64 (or FP32) range.  With mu = 1 and lambda = 1/2, across
the element along z
  P_zz = ln J,   dP_zz of du_z = z is 3 - ln J,   and the diagonal of a z-DoF of Q1 is
  (3 mu + mu + 2 lambda (1 - ln J)) / 9,
all ordinary numbers, while A = J F^-1 and J^2 are near or beyond the range."""
import numpy as np
import pytest

from tests.gpu_util import cuda, host, lib_or_fail

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
FP64 = [(3.0, 5.0), (1e70, 1e70), (1e76, 1e76), (1e80, 1e81), (1e100, 1e120), (1e154, 1e140), (1e154, 6e153),
        (9e153, 9e153), (1.2e154, 1e154)]   # the last three are above 0.75 * 2^1022 and 0.75 * 2^1023
FP32 = [(3.0, 5.0), (1e8, 1e8), (1e9, 2e9), (1e10, 1e10), (1e15, 1e16), (1e18, 1e18), (1e19, 2e18)]


def nodes(p):
    """Reference coordinates of the nodes of a line: Gauss-Lobatto points on [0, 1]."""
    return {1: [0.0, 1.0], 2: [0.0, 0.5, 1.0], 3: [0.0, 0.5 - np.sqrt(0.05), 0.5 + np.sqrt(0.05), 1.0],
            4: [0.0, 0.5 - np.sqrt(3 / 28), 0.5, 0.5 + np.sqrt(3 / 28), 1.0]}[p]


def state(p, a, b):
    t = np.array(nodes(p))
    n = p + 1
    u = np.zeros((3, n, n, n))
    u[0] = a * t[None, None, :]
    u[1] = b * t[None, :, None]
    du = np.zeros((3, n, n, n))
    du[2] = t[:, None, None]
    ln = float(np.log1p(np.longdouble(a)) + np.log1p(np.longdouble(b)))
    return u.reshape(-1), du.reshape(-1), ln


def top(v, p):
    return v.reshape(3, p + 1, p + 1, p + 1)[2, -1].sum()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("a,b", FP64)
def test_fp64(p, a, b):
    import torch
    nhmf = lib_or_fail()
    u, du, ln = state(p, a, b)
    # ln J takes the gradients' roundings (16 units of a and of b), the sums a few units of each term
    # per pass (up to 25 products of coefficients below 10) against |3 - ln J| and |ln J| above 0.2
    tol = 4096 * U * (3 + abs(ln))
    prob = nhmf.Problem(1, p, 1.0, 0.5, nhmf.NHMF_BC_NONE)
    ut, dut = cuda(u), cuda(du)
    prob.set_linearization(ut, 0)
    got = host(prob.apply(dut, torch.empty_like(dut), nhmf.NHMF_FP64, nhmf.NHMF_ON_THE_FLY))
    assert abs(top(got, p) - (3.0 - ln)) <= tol, ("on the fly", top(got, p), 3.0 - ln)
    got = host(prob.residual(ut, torch.empty_like(dut)))
    assert abs(top(got, p) - ln) <= tol, ("residual", top(got, p), ln)
    d_fly = host(prob.diagonal(torch.empty_like(dut)))
    prob.set_linearization(ut, nhmf.NHMF_CACHE_FP64)
    got = host(prob.apply(dut, torch.empty_like(dut), nhmf.NHMF_FP64, nhmf.NHMF_CACHED))
    assert abs(top(got, p) - (3.0 - ln)) <= tol, ("cached", top(got, p), 3.0 - ln)
    d_cached = host(prob.diagonal(torch.empty_like(dut)))
    if p == 1:
        for d in (d_fly, d_cached):
            assert np.abs(d[16:] - (5.0 - ln) / 9.0).max() <= tol, (d[16:], (5.0 - ln) / 9.0)
    prob.close()


@pytest.mark.parametrize("p", [1, 2, 3, 4])
@pytest.mark.parametrize("a,b", FP32)
def test_fp32(p, a, b):
    import torch
    nhmf = lib_or_fail()
    u, du, ln = state(p, a, b)
    prob = nhmf.Problem(1, p, 1.0, 0.5, nhmf.NHMF_BC_NONE)
    dut = cuda(du).float()
    tol = 4096 * 2.0 ** -24 * (3 + abs(ln))   # as above, in FP32's units
    for mask, strat in ((0, nhmf.NHMF_ON_THE_FLY), (nhmf.NHMF_CACHE_FP32, nhmf.NHMF_CACHED)):
        prob.set_linearization(cuda(u), mask)
        got = host(prob.apply(dut, torch.empty_like(dut), nhmf.NHMF_FP32, strat))
        assert abs(top(got, p) - (3.0 - ln)) <= tol, (strat, top(got, p), 3.0 - ln)
    prob.close()
