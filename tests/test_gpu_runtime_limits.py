"""What the library asks of the CUDA runtime, seen by a small shared object that is
preloaded into a child process and passes the calls on.  The shared-memory limit
of a kernel is an attribute of the function, not of a launch: contexts of different
width must set the same value, or one thread's value comes between another's and
its launch.  A launch whose CTAs must all be resident may be refused (part of the
GPU given to others): Lanczos steps and entanglement spectra then take the kernels
that need no such thing, and so they do when such a launch's wait for its CTAs ran
out (the shim sets the flag that the kernel sets then, and launches nothing)."""
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


def _child(tmp_path, shim, code, include=None):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, so = tmp_path / "shim.c", tmp_path / "shim.so"
    src.write_text(shim)
    inc = ["-I", include] if include else []
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", *inc, "-o", str(so), str(src), "-ldl"], check=True)
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


REFUSE = r"""
#define _GNU_SOURCE
#include <cuda_runtime_api.h>
#include <dlfcn.h>
#include <stdio.h>
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* cfg, const void* f, void** args) {
  static cudaError_t (*real)(const cudaLaunchConfig_t*, const void*, void**);
  if (!real) real = (cudaError_t(*)(const cudaLaunchConfig_t*, const void*, void**))dlsym(RTLD_NEXT, "cudaLaunchKernelExC");
  for (unsigned i = 0; i < cfg->numAttrs; ++i)
    if (cfg->attrs[i].id == cudaLaunchAttributeCooperative && cfg->attrs[i].val.cooperative) {
      fprintf(stderr, "REFUSED\n");
      return cudaErrorCooperativeLaunchTooLarge;
    }
  return real(cfg, f, args);
}
"""

RUN = """
import json, numpy as np, torch, workloads as W, paper_2605_07621_gb300 as ed
out = {}
c = ed.build_local_ops(ed.build_sectors(W.hubbard_chain(11, 1.0, 4.0, 5, 5)))
v = W.start_values(c.state_keys())
v = torch.tensor(v / np.linalg.norm(v), device="cuda")
for mode in ("f64", "f32"):
    r = ed.lanczos_ground(c, mode, max_iter=14, fixed_iter=True, v0=v)
    out[mode] = [r.alpha.tolist(), r.beta.tolist()]
for n in (4, 6):
    c = ed.build_sectors(W.hubbard_chain(2 * n, 1.0, 4.0, n, n))
    m = int(round(c.dim ** 0.5))
    psi = np.random.default_rng(n).standard_normal((m, m))
    psi /= np.linalg.norm(psi)
    lam = ed.entanglement_spectrum(c, torch.tensor(psi.ravel(), device="cuda")).lam[0]
    ref = np.linalg.svd(psi, compute_uv=False) ** 2
    assert np.abs(lam - ref).max() <= 1e-12, np.abs(lam - ref).max()
print("OUT", json.dumps(out))
"""


LATE = REFUSE.replace("""      fprintf(stderr, "REFUSED\\n");
      return cudaErrorCooperativeLaunchTooLarge;
""", """      /* the error flag is the last parameter: of the step (no dynamic shared memory) the 17th, of the panel the 12th */
      static int seen[2];
      const int panel = cfg->dynamicSmemBytes > 0;
      if (seen[panel]++ != 3) continue;
      fprintf(stderr, "LATE %d\\n", panel);
      return cudaMemsetAsync(*(void**)args[panel ? 11 : 16], 4, 1, cfg->stream);
""")


@pytest.mark.parametrize("what", ["REFUSED", "LATE"])
def test_cooperative_launch(tmp_path, what):
    import json

    import numpy as np

    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    shim = REFUSE if what == "REFUSED" else LATE
    shims = (shim, shim.replace(" && cfg->attrs[i].val", " && 0 && cfg->attrs[i].val"))  # the second passes all on
    rs = [_child(tmp_path, x, RUN, inc) for x in shims]
    assert rs[0].stderr.count(what) >= (4 if what == "REFUSED" else 2) and what not in rs[1].stderr
    runs = [json.loads(r.stdout.split("OUT", 1)[1]) for r in rs]
    for mode, tol in (("f64", 1e-11), ("f32", 2e-5)):  # as in test_gpu_lanczos_step
        (a, b), (a0, b0) = (np.array(r[mode]) for r in runs)
        scale = np.abs(a0).max() + np.abs(b0).max()
        assert np.abs(a - a0)[:12].max() <= tol * scale and np.abs(b - b0)[:12].max() <= tol * scale
