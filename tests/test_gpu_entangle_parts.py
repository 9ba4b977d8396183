"""Entanglement spectra whose tridiagonal matrices fall apart: blocks without
weight (exact zeros, at any norm of the state), product states and Schmidt-diagonal
ones with amplitudes 2^-k over 20 decades of the levels (a part per row, and every
digit exact: exact levels), and blocks made of
independent pieces of 1 to 700 rows, the second half of them scaled by 1e-4 (each
piece's levels to 1e-12 of its own largest, the bound that test_gpu_entangle_panel
derives for a whole block)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ed():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    return ed


@pytest.mark.parametrize("norm", [1.0, 1e-12])
def test_blocks_without_weight(ed, norm):
    import torch

    ctx = ed.build_sectors(W.j1j2_torus(4, 4, cut_mask=0xFF))
    _, dA, dB, _ = ctx.blocks()
    off, q = np.concatenate([[0], np.cumsum(dA * dB)]), len(dA) // 2
    psi = np.random.default_rng(3).standard_normal((int(dA[q]), int(dB[q])))
    psi *= norm / np.linalg.norm(psi)
    x = np.zeros(ctx.dim)
    x[off[q]:off[q + 1]] = psi.ravel()
    es = ed.entanglement_spectrum(ctx, torch.tensor(x, device="cuda"))
    ref = np.linalg.svd(psi, compute_uv=False) ** 2
    assert all(not np.any(lam) for i, lam in enumerate(es.lam) if i != q)
    assert np.abs(es.lam[q] - ref).max() <= 1e-12 * norm ** 2
    p = ref / ref.sum()
    assert abs(es.entropy + (p * np.log(p)).sum()) <= 1e-10


def test_product_state(ed):
    import torch

    ctx = ed.build_sectors(W.j1j2_torus(4, 4, cut_mask=0xFF))
    x = torch.zeros(ctx.dim, device="cuda", dtype=torch.float64)
    x[ctx.dim // 2 + 123] = 1.0
    es = ed.entanglement_spectrum(ctx, x)
    lam = np.concatenate(es.lam)
    assert np.count_nonzero(lam) == 1 and lam.max() == 1.0 and es.entropy == 0.0


@pytest.mark.parametrize("L,n", [(4, 2), (8, 4), (12, 5), (13, 6)])
def test_schmidt_diagonal(ed, L, n):
    import torch

    ctx = ed.build_sectors(W.hubbard_chain(L, 1.0, 4.0, n, n))
    m = int(round(ctx.dim ** 0.5))
    x = np.diag(0.5 ** np.random.default_rng(m).integers(0, 34, m))
    es = ed.entanglement_spectrum(ctx, torch.tensor(x.ravel(), device="cuda"))
    assert np.array_equal(es.lam[0], np.sort(np.diag(x) ** 2)[::-1])


@pytest.mark.parametrize("L,n,sizes", [(4, 2, [1, 2, 3]), (9, 4, [40, 1, 1, 84]), (13, 6, [1, 300, 63, 1, 700, 65, 2, 584])])
def test_independent_pieces(ed, L, n, sizes):
    import torch

    ctx = ed.build_sectors(W.hubbard_chain(L, 1.0, 4.0, n, n))
    rng = np.random.default_rng(sum(sizes))
    psi, at, ref, tol = np.zeros((sum(sizes),) * 2), 0, [], []
    assert psi.size == ctx.dim
    for i, k in enumerate(sizes):
        b = rng.standard_normal((k, k)) * (1e-4 if 2 * i >= len(sizes) else 1.0) / sum(sizes)
        psi[at:at + k, at:at + k] = b
        at += k
        s = np.linalg.svd(b, compute_uv=False) ** 2
        ref.append(s)
        tol.append(np.full(k, 1e-12 * s[0]))
    ref, tol = np.concatenate(ref), np.concatenate(tol)
    o = np.argsort(-ref, kind="stable")
    es = ed.entanglement_spectrum(ctx, torch.tensor(psi.ravel(), device="cuda"))
    assert (np.diff(es.lam[0]) <= 0).all()
    # levels of the two scales interleave: each within the larger bound of its neighbours at that rank
    d, t = np.abs(es.lam[0] - ref[o]), tol[o]
    t = np.maximum(t, np.maximum(np.append(t[1:], 0.0), np.insert(t[:-1], 0, 0.0)))
    assert (d <= t).all(), (d / t).max()
