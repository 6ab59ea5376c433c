"""The bias gradient of a stride-1 layer sums each block's voxels in nine FP32 chains: one voxel far
larger than the others costs the sum only what follows it in its own chain.

The network is zero but for the identity taps that carry the loss's gradient to layer t0.  That is
2^26 s at the first voxel and s at every other one: behind the large value a chain drops the s's
(they arrive four at a time, half a unit of 2^26 s).  A block holds at most 900 chunks of 16
positions, of which a lane sums 4 (units of the 193^3 grid spread over 608 blocks); beside the ninth
that is lost, adding the large sum to the other sums rounds to a multiple of 8 s at most 90 times."""
import numpy as np
import pytest

from oracle import unet as ounet
from tests.gpu_util import cuda, lib_or_fail
from tests.unet_cases import flat_params, unflat

pytestmark = pytest.mark.gpu


def test_large_voxel_costs_a_ninth():
    import torch
    nhmf = lib_or_fail()
    n_el, M = 96, 193
    params = {}
    for name, kind, cin, cout in ounet.LAYERS:
        params[name + ".w"] = np.zeros(ounet.weight_shape(kind, cin, cout))
        params[name + ".b"] = np.zeros(cout)
    for c in range(3):
        params["out.w"][c, c, 1, 1, 1] = 1.0
        params["t0.b"][c] = 1.0      # active, so that the ReLU passes the gradient
        params["out.b"][c] = -1.0    # the output is zero
    prob = nhmf.Problem(n_el, 2, 1.0, 1.5, nhmf.NHMF_BC_NONE)
    nhmf.nhmf_unet_create(prob.ctx)
    nhmf.nhmf_unet_set_params(prob.ctx, flat_params(params))
    x = torch.zeros(3 * M ** 3, dtype=torch.float32, device="cuda:0")
    e = torch.zeros(3, M ** 3, dtype=torch.float32, device="cuda:0")
    e[0] = -1.0
    e[0, 0] = -2.0 ** 26
    _, g = nhmf.nhmf_unet_loss_grad(prob.ctx, x, e.reshape(-1))
    s = 2.0 ** -51    # 2 / sum e^2, rounded to FP32
    got = unflat(g.astype(np.float64))["t0.b"][0] / s
    want = 2.0 ** 26 + (M ** 3 - 1)
    assert abs(got - want) <= 4 * 900 / 9 + 4 * 90, got - want
    prob.close()
