"""Several multigrid contexts alive at once, each solved in turn: what one hierarchy sets on the
device leaves the others' launches as they are.  Coarsest meshes of 2^3, 3^3, 5^3, 9^3 and 13^3
elements: the coarse solve's shared memory differs between all of them and its cluster between the
larger ones."""
import threading

import pytest

import nhmf_inputs as inp
from tests.gpu_util import cuda, lib_or_fail

pytestmark = pytest.mark.gpu
SIZES = [(2, 6), (1, 13), (1, 9), (2, 10), (1, 8)]   # (degree, elements): coarsest 3, 13, 9, 5, 2


def make(nhmf, p, N):
    w = inp.Workload("two", N, p, 1.0, 1.5, 1, "scaled", 0.01, "normal", 1.0, 4700 + N, 4800 + N)
    prob = nhmf.Problem.from_workload(w)
    prob.set_linearization(cuda(inp.draw_u(w)), nhmf.NHMF_CACHE_FP64 | nhmf.NHMF_CACHE_FP32)
    return prob, cuda(inp.draw_du(w))


def solve(nhmf, prob, b, solver):
    import torch
    x = torch.empty_like(b)
    it, inner, rel = prob.linear_solve(b, x, solver=solver, linear_rtol=1e-9)
    assert rel <= 1.01e-9
    return x, it, inner


def test_solved_in_turn():
    import torch
    nhmf = lib_or_fail()
    cases = [make(nhmf, p, N) for p, N in SIZES]
    solvers = (nhmf.NHMF_SOLVER_GMG, nhmf.NHMF_SOLVER_MIXED_GMG)
    first = [[solve(nhmf, *c, s) for s in solvers] for c in cases]
    for order in (range(len(cases)), reversed(range(len(cases)))):
        for k in order:
            for s, want in zip(solvers, first[k]):
                x, it, inner = solve(nhmf, *cases[k], s)
                assert torch.equal(x, want[0]) and (it, inner) == want[1:]
    for prob, _ in cases:
        prob.close()


def test_two_host_threads():
    nhmf = lib_or_fail()
    errors = []

    def work(p, N):
        import torch
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                for _ in range(3):
                    prob, b = make(nhmf, p, N)   # a new hierarchy is set up while the other thread solves
                    for _ in range(5):
                        solve(nhmf, prob, b, nhmf.NHMF_SOLVER_MIXED_GMG)
                    prob.close()
        except Exception as e:   # reported by the test's own thread
            errors.append((p, N, e))

    threads = [threading.Thread(target=work, args=a) for a in ((2, 6), (1, 8))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
