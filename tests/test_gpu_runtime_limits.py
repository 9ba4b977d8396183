"""What the library asks of the CUDA runtime, seen by a small shared object that is
preloaded into a child process and passes the calls on.  The shared-memory limit
of a kernel is an attribute of the function, not of a launch: contexts of different
width must set the same value, or one thread's value comes between another's and
its launch."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
int cudaFuncSetAttribute(const void* f, int attr, int value) {
  static int (*real)(const void*, int, int);
  if (!real) real = (int (*)(const void*, int, int))dlsym(RTLD_NEXT, "cudaFuncSetAttribute");
  fprintf(stderr, "SETATTR %p %d %d\n", f, attr, value);
  return real(f, attr, value);
}
"""


def _child(tmp_path, shim, code):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, so = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(shim)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", str(so), str(src), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", code], cwd=ROOT, env=dict(os.environ, LD_PRELOAD=str(so)),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return r


WIDTHS = """
import numpy as np, torch, workloads as W, paper_2605_07621_gb300 as ed
def chain(nA, nB, k, spread):
    n = nA + nB
    J = 1.0 + (np.arange(n) * 0.37 % 1.0 if spread else np.zeros(n))
    return W.Model("spin", n, W.chain_bonds(n, True), jxy=list(J), jz=list(J), n_up=k, cut_mask=(1 << nA) - 1)
for spread in (False, True):  # five and more value classes: the general path
    for nB, k in ((12, 6), (11, 5), (14, 7), (15, 7), (16, 8), (15, 6)):
        c = ed.build_local_ops(ed.build_sectors(chain(1, nB, k, spread)))
        assert (c.row_pass(torch.float64) == "k_row5") != spread
        for dt in (torch.float64, torch.float32):
            x = torch.randn(c.dim + 1, device="cuda", dtype=dt)
            for v in (x[:-1], x[1:]):  # the second is not 16-byte aligned
                ed.apply_H(c, v, torch.empty_like(v))
torch.cuda.synchronize()
"""


def test_one_shared_memory_limit_per_kernel(tmp_path):
    r = _child(tmp_path, SHIM, WIDTHS)
    seen = {}
    for line in r.stderr.splitlines():
        if line.startswith("SETATTR"):
            _, f, attr, value = line.split()
            seen.setdefault((f, attr), set()).add(int(value))
    assert len(seen) >= 6
    assert all(len(v) == 1 for v in seen.values()), seen
