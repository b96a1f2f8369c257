"""A stage whose tensor map cannot be encoded is refused before any of its kernels is launched.

The map is the one thing in a stage that can be refused; on a working machine it never is. The
child process finds no driver entry for the encoding: a preloaded wrapper of the runtime's lookup
(compiled here with gcc) answers "not found" for that one name and passes every other on. The
refused call must return FWI_E_CUDA and must not have written the caller's device buffer, which a
kernel of the stage would have."""
import os
import shutil
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

WRAPPER = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <string.h>
typedef int (*lookup)(const char *, void **, unsigned, unsigned long long, int *);
int cudaGetDriverEntryPointByVersion(const char *name, void **fn, unsigned version, unsigned long long flags, int *found) {
  if (!strcmp(name, "cuTensorMapEncodeTiled")) {
    *fn = 0;
    if (found) *found = 1; /* cudaDriverEntryPointSymbolNotFound */
    return 0;
  }
  return ((lookup)dlsym(RTLD_NEXT, "cudaGetDriverEntryPointByVersion"))(name, fn, version, flags, found);
}
"""

CHILD = r"""
import numpy as np, torch
import fwi_inputs as fi
from paper_1504_08340_gb300 import Context, FWIError
w = fi.tiny(nx=3, ny=3, nz=2, npml=2, nsteps=4, f0=30.0, nrec_side=2)
lam, mu = (np.ascontiguousarray(a, dtype=np.float32) for a in fi.medium(w, "true"))
with Context(w.nx, w.ny, w.nz, w.npml, w.h, w.dt, w.nsteps, rho=w.rho) as ctx:
    ctx.set_material(lam, mu)
    n = ctx.state().size
    state = torch.zeros(n, dtype=torch.float32, device="cuda")
    rate = torch.full((n,), 7.0, dtype=torch.float32, device="cuda")
    for adjoint in (False, True):
        try:
            ctx.rhs(state, adjoint=adjoint, out=rate)
        except FWIError as e:
            assert e.name == "FWI_E_CUDA" and "tensor map" in str(e), e
        else:
            raise AssertionError("the stage was not refused")
        torch.cuda.synchronize()
        assert bool((rate == 7.0).all()), "a refused stage wrote the rate"
print("refused cleanly")
"""


def test_refused_stage_launches_nothing(tmp_path):
    gcc = shutil.which("gcc")
    if not gcc:
        pytest.skip("no gcc")
    src, lib = tmp_path / "wrap.c", tmp_path / "wrap.so"
    src.write_text(WRAPPER)
    subprocess.run([gcc, "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=ROOT)
    out = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=ROOT, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0 and "refused cleanly" in out.stdout, out.stdout + out.stderr
