"""A kernel's limit of dynamic shared memory belongs to the device: work on a small problem must not
lower it, or another host thread's launch for a larger problem fails in between.  A preloaded
cudaFuncSetAttribute counts the calls that lower a kernel's limit while networks and multigrid
hierarchies of different sizes run in turn."""
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
static const void* func[1024];
static int limit[1024], kernels, lowered, calls;
int limits_lowered(void) { return lowered; }
int limits_calls(void) { return calls; }
int cudaFuncSetAttribute(const void* f, int attr, int value) {
  if (attr == 8) {  /* cudaFuncAttributeMaxDynamicSharedMemorySize */
    int i = 0;
    ++calls;
    while (i < kernels && func[i] != f) ++i;
    if (i == kernels && kernels < 1024) { func[kernels] = f; limit[kernels++] = value; }
    else if (i < 1024) { lowered += value < limit[i]; limit[i] = value; }
  }
  int (*real)(const void*, int, int) = (int (*)(const void*, int, int))dlsym(RTLD_NEXT, "cudaFuncSetAttribute");
  return real(f, attr, value);
}
"""
CHILD = r"""
import ctypes, sys
import numpy as np
import torch
import nhmf_inputs as inp
from paper_2505_15535_gb300 import nhmf
from tests.unet_cases import flat_params, he_params
nets = []
for n in (48, 8):
    prob = nhmf.Problem(n, 2, 1.0, 1.5, nhmf.NHMF_BC_COMPRESSION)
    nhmf.nhmf_unet_create(prob.ctx)
    nhmf.nhmf_unet_set_params(prob.ctx, flat_params(he_params()))
    rng = np.random.default_rng(n)
    nets.append((prob, *(torch.from_numpy(rng.standard_normal(prob.n_dofs).astype(np.float32)).cuda() for _ in range(2))))
for _ in range(2):
    for prob, x, e in nets:
        nhmf.nhmf_unet_loss_grad(prob.ctx, x, e)
for p, N in ((2, 6), (1, 8), (3, 4), (1, 9)):
    w = inp.Workload("limits", N, p, 1.0, 1.5, 1, "scaled", 0.01, "normal", 1.0, 5401, 5402)
    prob = nhmf.Problem.from_workload(w)
    prob.set_linearization(torch.from_numpy(inp.draw_u(w)).cuda(), 3)
    b = torch.from_numpy(inp.draw_du(w)).cuda()
    for solver in (nhmf.NHMF_SOLVER_GMG, nhmf.NHMF_SOLVER_MIXED_GMG):
        prob.linear_solve(b, torch.empty_like(b), solver=solver)
L = ctypes.CDLL(sys.argv[1])
print(L.limits_calls(), L.limits_lowered())
"""


def test_no_call_lowers_a_limit(tmp_path):
    lib_or_fail()
    src, lib = tmp_path / "fake.c", tmp_path / "libfake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(lib), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD, str(lib)], env=env, cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    calls, lowered = (int(v) for v in r.stdout.split())
    assert calls > 0 and lowered == 0, (calls, lowered)
