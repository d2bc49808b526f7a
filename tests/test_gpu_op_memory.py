"""tm_op_create without the memory for the fixed-point copy of the FP64 links: the
operator works all the same, on the FP64 kernel.  The allocation fails on the
host, in a stand-in for the runtime's call that a child process loads before the
runtime."""
import os
import shutil
import subprocess
import sys

import pytest

from .gpu_util import require_gpu

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <stdlib.h>
int cudaMallocFromPoolAsync(void **p, size_t n, void *pool, void *s) {
  static int (*real)(void **, size_t, void *, void *);
  if (!real) real = (int (*)(void **, size_t, void *, void *))dlsym(RTLD_NEXT, "cudaMallocFromPoolAsync");
  if (n == strtoul(getenv("TM_TEST_FAIL_BYTES"), 0, 10)) {
    fputs("refused\n", stderr);
    return 2; /* cudaErrorMemoryAllocation */
  }
  return real(p, n, pool, s);
}
"""

CHILD = """
import numpy as np, torch
from oracle import operator as oop
from paper_1401_6749_gb300 import synth, tmloops as tl
from tests.gpu_util import pack, to_dev, unpack
L = (6, 4, 2, 10)
U = synth.gauge_field(L, 3)
op = tl.Operator(L, 0.16, 0.01, to_dev(U))
psi = synth.random_spinor(L, 3, 4)
f = pack(tl, L, psi, tl.F64)
out = torch.empty_like(f)
tl.tm_dslash(op, out, f, 3, prec=tl.F64)
got = unpack(tl, L, out, tl.F64, 3)
ref = oop.apply_M(U, psi, 0.16, 0.01)
assert np.linalg.norm(got - ref) <= 4e-16 * np.linalg.norm(ref)
print("child ok")
"""


def test_operator_without_fixed_point_links(tmp_path):
    require_gpu()
    if shutil.which("gcc") is None:
        pytest.skip("no C compiler")
    src, lib = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    sites = 6 * 4 * 2 * 10 // 2  # per parity; a ragged number of groups of 32, so no other copy has these bytes
    nbytes = 8 * ((sites + 31) // 32) * 288 * 16
    env = dict(os.environ, LD_PRELOAD=str(lib), TM_TEST_FAIL_BYTES=str(nbytes), PYTHONPATH=ROOT)
    run = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=600)
    assert run.returncode == 0, run.stderr[-2000:]
    assert "child ok" in run.stdout and "refused" in run.stderr
