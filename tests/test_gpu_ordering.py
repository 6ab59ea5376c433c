"""Launches that start while the one before them drains: FP32 applies (element kernel, then node
gather) whose input the stream has only just written and whose output it reads at once, and multigrid
cycles (smoothing, transfers), give bit by bit what they give with the GPU idle in between."""
import pytest

import nhmf_inputs as inp
from tests.gpu_util import cuda, lib_or_fail

pytestmark = pytest.mark.gpu


def problem(nhmf, p, N, amp=0.05):
    w = inp.Workload("order", N, p, 1.0, 1.5, 1, "scaled", amp, "normal", 1.0, 4300 + N, 4400 + N)
    prob = nhmf.Problem.from_workload(w)
    prob.set_linearization(cuda(inp.draw_u(w)), nhmf.NHMF_CACHE_FP64 | nhmf.NHMF_CACHE_FP32)
    return prob, cuda(inp.draw_du(w))


@pytest.mark.parametrize("strat", [0, 1])
@pytest.mark.parametrize("p,N", [(1, 9), (1, 40), (2, 12), (2, 64), (3, 11), (4, 10)])
def test_fp32_applies_back_to_back(p, N, strat):
    import torch
    nhmf = lib_or_fail()
    prob, d = problem(nhmf, p, N)
    d = d.float()
    want, x = [], d.clone()
    for _ in range(3):
        y = prob.apply(x, torch.empty_like(x), nhmf.NHMF_FP32, strat)
        torch.cuda.synchronize()
        want.append(y)
        x = 0.5 * y
    torch.cuda.synchronize()
    v = torch.empty_like(d)
    for _ in range(20):
        x = d
        for k in range(3):
            prob.apply(x, v, nhmf.NHMF_FP32, strat)   # the same output, and so the same scratch, each time
            y = v.clone()
            assert torch.equal(y, want[k])
            x = 0.5 * y
    # applies with nothing in between: each one's gather and the next one's element kernel share vloc
    outs = [torch.empty_like(d) for _ in range(12)]
    prob.apply(d, outs[0], nhmf.NHMF_FP32, strat)
    for a, b in zip(outs, outs[1:]):
        prob.apply(a, b, nhmf.NHMF_FP32, strat)
    torch.cuda.synchronize()
    x = d
    for out in outs:
        y = prob.apply(x, torch.empty_like(x), nhmf.NHMF_FP32, strat)
        torch.cuda.synchronize()
        assert torch.equal(y, out)
        x = out
    prob.close()


@pytest.mark.parametrize("p,N", [(1, 16), (2, 8), (3, 12)])
def test_multigrid_repeats(p, N):
    import torch
    nhmf = lib_or_fail()
    prob, b = problem(nhmf, p, N, 0.01)
    first = None
    for _ in range(6):
        x = torch.empty_like(b)
        it = prob.linear_solve(b, x, solver=nhmf.NHMF_SOLVER_MIXED_GMG, linear_rtol=1e-10)
        assert first is None or (torch.equal(x, first[0]) and it == first[1])
        first = first or (x, it)
    prob.close()


@pytest.mark.parametrize("solver", ["NHMF_SOLVER_JACOBI_CG", "NHMF_SOLVER_MIXED_GMG"])
def test_first_solve_beside_a_busy_default_stream(solver):
    """A context's first solve clears its reduction scratch and builds its hierarchy; on a side stream
    this is ordered although the default stream is still busy with something else."""
    import torch
    nhmf = lib_or_fail()
    results = []
    for busy in (False, True, True):
        prob, b = problem(nhmf, 2, 6, 0.01)
        x = torch.empty_like(b)
        side = torch.cuda.Stream()
        torch.cuda.synchronize()
        if busy:
            torch.cuda._sleep(400_000_000)   # about 0.2 s
        with torch.cuda.stream(side):
            it = prob.linear_solve(b, x, solver=getattr(nhmf, solver), linear_rtol=1e-10)
        torch.cuda.synchronize()
        results.append((it, x))
        prob.close()
    assert all(it == results[0][0] and torch.equal(x, results[0][1]) for it, x in results[1:])


@pytest.mark.parametrize("p,N", [(1, 9), (2, 6), (4, 5)])
def test_applies_in_a_callers_capture(p, N):
    """A caller's captured stream may hold anything before an apply: a copy, a memset, an event of
    another stream.  The graph replays with the inputs of the moment."""
    import torch
    nhmf = lib_or_fail()
    prob, d = problem(nhmf, p, N)
    for prec, dt in ((nhmf.NHMF_FP64, torch.float64), (nhmf.NHMF_FP32, torch.float32)):
        src = d.to(dt)
        x, v, y, z = (torch.empty_like(src) for _ in range(4))
        prob.apply(src, v, prec, 1)   # every kernel is loaded
        torch.cuda.synchronize()
        graph, side = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph):
            x.copy_(src)
            prob.apply(x, v, prec, 1)      # behind a copy
            y.zero_()
            prob.apply(v, y, prec, 0)      # behind a memset of its own output
            cur = torch.cuda.current_stream()
            side.wait_stream(cur)
            with torch.cuda.stream(side):
                z.copy_(y)
            cur.wait_stream(side)
            prob.apply(z, v, prec, 1)      # behind another stream's event
        for scale in (1.0, -2.0):
            src.copy_(scale * d.to(dt))
            graph.replay()
            torch.cuda.synchronize()
            a = prob.apply(src, torch.empty_like(src), prec, 1)
            b = prob.apply(a, torch.empty_like(src), prec, 0)
            c = prob.apply(b, torch.empty_like(src), prec, 1)
            torch.cuda.synchronize()
            assert torch.equal(y, b) and torch.equal(v, c), (prec, scale)
    prob.close()
