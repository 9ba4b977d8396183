"""Orthogonality that the re-orthogonalisation leaves: w against m orthonormal
vectors V (rows of ragged length, an FP32 plane beside them), called below the
C ABI.  max |<V_j, w>| <= 16 * 2^-53 |w| for coefficients at rounding level, for
ones too many and too large for the FP32 plane, for w almost inside the span (the
first pass leaves 1e-12 of it: the second pass's coefficients are then 1e-4 of what
is left) and without a plane.  The bound: the update's own rounding is a vector
of norm at most 2^-53 |w| and the plane's at most half of that, and a dot product
of 10,007 terms in FP64 adds some 2^-53 |w|.  And the w that is left agrees with
(I - V V^T) w in FP64 to 1e-13 of the input's norm."""
import ctypes

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

CASES = {"rounding": (1e-15, 1.0, True), "single_1e-9": (1e-9, 1.0, True), "at_2^-37": (2.0 ** -37, 1.0, True),
         "inside": (1.0, 1e-12, True), "ordinary": (1.0, 1.0, True), "no_plane": (1e-15, 1.0, False)}


@pytest.mark.parametrize("m", [1, 7, 8, 300])
@pytest.mark.parametrize("name", list(CASES))
def test_orthogonality(name, m):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed
    from paper_2605_07621_gb300 import _lib

    n = 10007
    coef, rest, plane = CASES[name]
    rng = np.random.default_rng(m)
    Q = np.linalg.qr(rng.standard_normal((n, m + 1)))[0].T
    h = coef * rng.uniform(0.5, 1.0, m) * rng.choice([-1.0, 1.0], m)
    if name.startswith("single"):
        h[1:] *= 1e-7
    w0 = h @ Q[:m] + rest * Q[m]
    V = torch.tensor(np.ascontiguousarray(Q[:m]), device="cuda")
    w = torch.tensor(w0, device="cuda")

    ctx = ed.build_local_ops(ed.build_sectors(W.hubbard_chain(4, 1.0, 4.0, 2, 2)))
    lib = ctypes.CDLL(_lib.LIB_PATH)
    p, i, ll = ctypes.c_void_p, ctypes.c_int, ctypes.c_longlong
    f = {"ensure_scratch": ("_ZN3edk14ensure_scratchEP6ed_ctx", i, [p]),
         "slot": ("_ZN3edk4slotEP6ed_ctxi", p, [p, i]),
         "dot": ("_ZN3edk7dot_devIdEE9ed_statusP6ed_ctxPKT_S6_xPdP11CUstream_sti", i, [p, p, p, ll, p, p, i]),
         "read": ("_ZN3edk12read_scalarsEP6ed_ctxiiPdP11CUstream_st", i, [p, i, i, p, p]),
         "reorth": ("_ZN3edk15launch_reorth64EP6ed_ctxPKdPKfiPdxS6_P11CUstream_st", i, [p, p, p, i, p, ll, p, p]),
         "doubles": ("_ZN3edk16reorth64_doublesEi", ll, [i]), "ld": ("_ZN3edk7fp32_ldEx", ll, [ll])}
    for k, (sym, res, args) in f.items():
        fn = getattr(lib, sym)
        fn.restype, fn.argtypes = res, args
        f[k] = fn
    F = torch.zeros(m, f["ld"](n), device="cuda", dtype=torch.float32)
    F[:, :n] = V
    scratch = torch.empty(f["doubles"](m), device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    c, beta = ctx.handle, ctypes.c_double()
    assert f["ensure_scratch"](c) == 0
    assert f["dot"](c, w.data_ptr(), w.data_ptr(), n, f["slot"](c, 1), None, 1) == 0
    assert f["reorth"](c, V.data_ptr(), F.data_ptr() if plane else None, m, w.data_ptr(), n, scratch.data_ptr(), None) == 0
    assert f["read"](c, 1, 1, ctypes.addressof(beta), None) == 0
    nw = float(torch.linalg.vector_norm(w))
    assert abs(beta.value - nw) <= 1e-12 * nw
    assert float((V @ w).abs().max()) <= 16 * 2.0 ** -53 * nw
    ref = torch.tensor(w0, device="cuda")
    for _ in range(2):
        ref = ref - V.T @ (V @ ref)
    assert float(torch.linalg.vector_norm(w - ref)) <= 1e-13 * np.linalg.norm(w0)
