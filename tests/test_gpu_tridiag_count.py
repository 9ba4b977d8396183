"""The tridiagonal eigenvalues by counting on the GPU, through the entanglement
spectrum of states whose spectrum is known in closed form: diagonal blocks
(nothing to reduce: the eigenvalues are the squares of the diagonal) with
distinct levels, with a few multiplets of equal ones, with 16 decades between
them and with one level among zeros; one level in all; and many small blocks at
once next to large ones, which change the lanes per eigenvalue.  To 2.5e-14 of
the largest eigenvalue where the block is diagonal (48-bit digits of the Gram
matrix's factors: 2^-46; the reduction's copy: 2^-47; the counts: 2^-52), and
with the sum of the levels equal to the block's weight to 1e-13."""
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


@pytest.mark.parametrize("kind", ["distinct", "multiplets", "decades", "one"])
@pytest.mark.parametrize("L,n", [(4, 4), (4, 2), (5, 2), (8, 4), (11, 5), (12, 6)])
def test_diagonal_blocks(ed, L, n, kind):
    import torch

    ctx = ed.build_sectors(W.hubbard_chain(L, 1.0, 4.0, n, n))
    m = int(round(ctx.dim ** 0.5))
    rng = np.random.default_rng(m)
    lam = {"distinct": rng.random(m), "multiplets": rng.integers(1, 4, m) / 4.0,
           "decades": np.logspace(0, -16, m), "one": np.eye(1, m, m // 2)[0]}[kind]
    x = np.diag(np.sqrt(lam))
    es = ed.entanglement_spectrum(ctx, torch.tensor(x.ravel(), device="cuda"))
    ref = np.sort(np.diag(x) ** 2)[::-1]
    assert np.abs(es.lam[0] - ref).max() <= 2.5e-14 * ref[0]
    assert (np.diff(es.lam[0]) <= 0).all()


@pytest.mark.parametrize("mask", [0x3F, 0xFFF, 0x7FFFFF, 0xFFFFFF])
def test_many_blocks(ed, mask):
    import torch

    ctx = ed.build_sectors(W.j1j2_torus(4, 6, cut_mask=mask))
    g = torch.Generator(device="cuda")
    g.manual_seed(mask)
    x = torch.randn(ctx.dim, device="cuda", dtype=torch.float64, generator=g)
    x /= x.norm()
    es = ed.entanglement_spectrum(ctx, x)
    s, dA, dB, _ = ctx.blocks()
    off = 0
    for lam, w, a, b in zip(es.lam, es.weight, dA, dB):
        blk = x[off:off + a * b].reshape(a, b)
        off += a * b
        assert abs(lam.sum() - w) <= 1e-13
        ref = torch.linalg.svdvals(blk.cpu()).numpy() ** 2
        assert np.abs(lam - ref).max() <= 1e-12
