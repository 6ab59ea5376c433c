"""The colour-chained FP64 and double-float kernels on both sides of the line between small and
normal blocks (152 SMs: Q1 26^3, Q2 25^3, Q3 16^3, Q4 12^3 elements; the diagonal's lies lower),
with ragged colour classes, on sampled oracle rows; and their ordering on streams."""
import numpy as np
import pytest

import nhmf_inputs as inp
from oracle.fem import Operator
from oracle.mesh import Mesh
from tests.gpu_util import cuda, host, lib_or_fail

pytestmark = pytest.mark.gpu


def workload(p, N, bc):
    return inp.Workload("shape", N, p, 1.0, 1.5, bc, "scaled", 0.05, "normal", 1.0, 4100 + N, 4200 + N)


@pytest.mark.parametrize("p,N,bc", [(1, 26, 2), (1, 27, 1), (2, 19, 0), (2, 25, 1), (2, 26, 2), (3, 13, 2), (3, 16, 1),
                                    (3, 17, 0), (4, 9, 1), (4, 12, 2), (4, 13, 2)])
def test_block_shapes(p, N, bc):
    import torch
    nhmf = lib_or_fail()
    w = workload(p, N, bc)
    u, du, fac = inp.draw_u(w), inp.draw_du(w), inp.inclusion_factors(N)
    du[inp.dirichlet_mask(N, p, bc).reshape(-1)] = 0.25  # identity rows show
    op = Operator(Mesh(N, p), 1.0, 1.5, bc, factors=fac)
    rows = np.unique(np.concatenate([np.random.default_rng(3).choice(w.n_dofs, 150, replace=False),
                                     [0, w.n_dofs - 1, w.n_dofs // 2]]))
    idx = torch.from_numpy(rows).to("cuda:0")
    prob = nhmf.Problem.from_workload(w)
    nhmf.nhmf_set_material_factors(prob.ctx, cuda(fac))
    prob.set_linearization(cuda(u), 15)
    dut = cuda(du)
    ref = op.apply_rows(u, du, rows)

    def check(v, want):
        assert np.linalg.norm(host(v[idx]) - want) <= 1e-12 * np.linalg.norm(want)

    for prec, strat in ((0, 0), (0, 1), (0, 2), (2, 1)):
        check(prob.apply(dut, torch.full_like(dut, np.nan), prec, strat), ref)
    check(prob.residual(cuda(u), torch.full_like(dut, np.nan)), op.residual_rows(u, rows))
    diag = op.diagonal_rows(u, rows)
    check(prob.diagonal(torch.full_like(dut, np.nan)), diag)   # from the point cache
    prob.set_linearization(cuda(u), 0)
    check(prob.diagonal(torch.full_like(dut, np.nan)), diag)   # from u
    prob.close()


@pytest.mark.parametrize("p,N", [(1, 8), (2, 12), (2, 30)])
def test_chain_ordering(p, N):
    """Applies whose input the stream has only just written and whose output it reads at once, and
    one context used from two streams in turn, give what separate applies give, bit by bit."""
    import torch
    nhmf = lib_or_fail()
    w = workload(p, N, 1)
    prob = nhmf.Problem.from_workload(w)
    prob.set_linearization(cuda(inp.draw_u(w)), nhmf.NHMF_CACHE_FP64)
    d0 = cuda(inp.draw_du(w))
    want, x = [], d0.clone()
    for _ in range(3):
        y = prob.apply(x, torch.empty_like(x), 0, 1)
        torch.cuda.synchronize()
        want.append(y)
        x = 0.5 * y
    for _ in range(20):
        x = d0.clone()
        for k in range(3):
            y = prob.apply(x, torch.empty_like(x), 0, 1)
            assert torch.equal(y, want[k])
            x = 0.5 * y
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    outs = []
    for k in range(20):
        with torch.cuda.stream(streams[k % 2]):
            outs.append(prob.apply(d0, torch.empty_like(d0), 0, 1))
    torch.cuda.synchronize()
    assert all(torch.equal(o, want[0]) for o in outs)
    prob.close()


@pytest.mark.parametrize("p,N", [(1, 5), (2, 1), (2, 5), (2, 7), (3, 2), (3, 3), (4, 1), (4, 3)])
@pytest.mark.parametrize("bc,model", [(0, 0), (1, 1), (2, 0)])
def test_fp32_column_kernel(p, N, bc, model):
    """FP32 applies on meshes that leave a block's last elements absent, with inclusions, both models
    and strategies; values on constrained DoFs, even NaN, reach no other row."""
    import torch
    nhmf = lib_or_fail()
    w = workload(p, N, bc)
    u, du, fac = inp.draw_u(w), inp.draw_du(w), inp.inclusion_factors(N, 10.0)
    op = Operator(Mesh(N, p), 1.0, 1.5, bc, model=model, factors=fac)
    ref = op.apply(u, du)
    fixed = inp.dirichlet_mask(N, p, bc).reshape(-1)
    du[fixed] = np.nan
    prob = nhmf.Problem(N, p, 1.0, 1.5, bc, model=model)
    nhmf.nhmf_set_material_factors(prob.ctx, cuda(fac))
    prob.set_linearization(cuda(u), 0 if model else nhmf.NHMF_CACHE_FP32)
    dut = cuda(du).float()
    for strat in (0,) if model else (0, 1):
        v = host(prob.apply(dut, torch.full_like(dut, 7.0), nhmf.NHMF_FP32, strat))
        assert np.isnan(v[fixed]).all()
        free = ~fixed
        assert np.linalg.norm(v[free] - ref[free]) <= 1e-5 * np.linalg.norm(ref[free])
    prob.close()


@pytest.mark.parametrize("N", [1, 3, 4, 15, 17])
@pytest.mark.parametrize("bc,model", [(0, 0), (1, 1), (2, 0)])
def test_fp32_register_kernel_q1(N, bc, model):
    """Q1 FP32 applies on meshes of less than one warp of elements up to several blocks, most of
    them not a multiple of a tile; with inclusions, both models and strategies."""
    import torch
    nhmf = lib_or_fail()
    w = workload(1, N, bc)
    u, du, fac = inp.draw_u(w), inp.draw_du(w), inp.inclusion_factors(N, 10.0)
    fixed = inp.dirichlet_mask(N, 1, bc).reshape(-1)
    du[fixed] = 0.25  # identity rows show
    ref = Operator(Mesh(N, 1), 1.0, 1.5, bc, model=model, factors=fac).apply(u, du)
    prob = nhmf.Problem(N, 1, 1.0, 1.5, bc, model=model)
    nhmf.nhmf_set_material_factors(prob.ctx, cuda(fac))
    prob.set_linearization(cuda(u), 0 if model else nhmf.NHMF_CACHE_FP32)
    dut = cuda(du).float()
    for strat in (0,) if model else (0, 1):
        v = host(prob.apply(dut, torch.full_like(dut, np.nan), nhmf.NHMF_FP32, strat))
        assert np.linalg.norm(v - ref) <= 1e-5 * np.linalg.norm(ref)
    prob.close()
