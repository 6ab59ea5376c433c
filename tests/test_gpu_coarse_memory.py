"""A device without room for the coarsest level's matrix: the solve runs as it does without one.  The
refusal is a fake cudaMalloc, preloaded into a child process, that answers one size with
cudaErrorMemoryAllocation."""
import os
import subprocess
import sys

import pytest

from tests.conftest import ROOT
from tests.gpu_util import lib_or_fail

pytestmark = pytest.mark.gpu

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
static unsigned refused;
unsigned fake_refused(void) { return refused; }
int cudaMalloc(void** p, size_t n) {
  const char* s = getenv("FAKE_REFUSE_BYTES");
  if (s && strtoull(s, 0, 10) == n) { ++refused; *p = 0; return 2; }
  int (*real)(void**, size_t) = (int (*)(void**, size_t))dlsym(RTLD_NEXT, "cudaMalloc");
  return real(p, n);
}
"""
CHILD = r"""
import ctypes, sys
import torch
import nhmf_inputs as inp
from paper_2505_15535_gb300 import nhmf
w = inp.Workload("memory", 8, 1, 1.0, 1.5, 1, "scaled", 0.01, "normal", 1.0, 5301, 5302)
prob = nhmf.Problem.from_workload(w)
prob.set_linearization(torch.from_numpy(inp.draw_u(w)).cuda(), 3)
b = torch.from_numpy(inp.draw_du(w)).cuda()
x = torch.empty_like(b)
its = []
for solver in (nhmf.NHMF_SOLVER_GMG, nhmf.NHMF_SOLVER_MIXED_GMG):
    it, inner, rel = prob.linear_solve(b, x, solver=solver, linear_rtol=1e-9)
    assert rel <= 1.01e-9
    its.append(it)
print(ctypes.CDLL(sys.argv[1]).fake_refused(), *its)
"""


def test_refused_matrix(tmp_path):
    lib_or_fail()
    src, lib = tmp_path / "fake.c", tmp_path / "libfake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    got = {}
    # the matrices of a coarsest mesh of 2^3 elements: elements', FP64 rows, FP32 rows
    for size in (0, 8 * 576 * 8, 81 * 104 * 8, 81 * 104 * 4):
        env = dict(os.environ, LD_PRELOAD=str(lib), FAKE_REFUSE_BYTES=str(size), PYTHONPATH=ROOT)
        r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], env=env, cwd=ROOT, capture_output=True, text=True,
                           timeout=300)
        assert r.returncode == 0, r.stderr[-2000:]
        got[size] = [int(v) for v in r.stdout.split()]
    assert got[0][0] == 0
    for size in list(got)[1:]:
        assert got[size][0] == 1, got           # asked for once, and refused
        assert abs(got[size][1] - got[0][1]) <= 1 and abs(got[size][2] - got[0][2]) <= 1, got
