"""The FP64 logarithm and reciprocal of the point code over their range, through the residual of one
Q1 element stretched by u_x = a x: with mu -> 0 and lambda = 1/2 the stress is P_yy = ln(1 + a) and
P_xx = ln(1 + a) / (1 + a), and the face sums of the nodal residual are these numbers."""
import numpy as np
import pytest

from tests.gpu_util import cuda, host, lib_or_fail

pytestmark = pytest.mark.gpu
U = 2.0 ** -53


def stretches():
    near_one = np.concatenate([s * 10.0 ** np.arange(-26, -2, 2) for s in (1.0, -1.0)])
    # table intervals (2^-8 below 1, 2^-7 above), their edges, and the octaves around them
    edges = np.concatenate([0.75 + np.arange(0, 64) / 256.0, 1.0 + np.arange(0, 64) / 128.0]) - 1.0
    edges = np.concatenate([edges, np.nextafter(edges, -1.0), edges + 1.0 / 512])
    wide = np.concatenate([2.0 ** np.arange(-9, 60, 3) * f - 1.0 for f in (0.75, 1.0, 1.4999)])
    a = np.concatenate([near_one, edges, wide])
    return np.unique(a[np.abs(a) >= 1e-26])


def test_log_and_reciprocal():
    import torch
    nhmf = lib_or_fail()
    prob = nhmf.Problem(1, 1, 1e-30, 0.5, nhmf.NHMF_BC_NONE)
    r = torch.empty(24, dtype=torch.float64, device="cuda:0")
    for a in stretches():
        u = np.zeros((3, 2, 2, 2))
        u[0, :, :, 1] = a
        got = host(prob.residual(cuda(u.reshape(-1)), r)).reshape(3, 2, 2, 2)
        with np.errstate(divide="ignore"):
            ln = float(np.log1p(np.longdouble(a)))
        # the gradient's rounding (four products and three sums) reaches ln J as dH / (1 + a), and
        # the function and the transposed sums a few units each
        tol = U * (16 + 16 * abs(a) / ((1 + a) * abs(ln)))
        assert abs(got[1, :, 1].sum() - ln) <= tol * abs(ln), (a, got[1, :, 1].sum(), ln)
        tol += U * (8 + 16 * abs(a) / (1 + a))
        pxx = 1e-30 * (1 + a) + (ln - 1e-30) / (1 + a)
        assert abs(got[0, :, :, 1].sum() - pxx) <= tol * abs(pxx), a
    for a, name in ((-1.0, "NONPOS_J"), (-1.5, "NONPOS_J"), (np.nan, "NONFINITE"), (np.inf, "NONFINITE")):
        u = np.zeros((3, 2, 2, 2))
        u[0, :, :, 1] = a
        with pytest.raises(nhmf.NhmfError, match=name):
            prob.residual(cuda(u.reshape(-1)), r)
    prob.close()
