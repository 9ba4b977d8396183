"""Reductions that take the three kernels per column, and that change to one launch
per panel on the way: one block of 6,435 rows (its first panels have more than
6,144), and 30 sites with 12 up spins, whose blocks of 3,003 rows share the
SMs with others and get fewer (16 of 152) than their first panels need (17).  Against the
eigenvalues of the block's Gram matrix in FP64.  The reduction's entries carry 48
bits, so a column adds at most 2^-48 of the largest eigenvalue, m columns m times
that.  Only blocks of more than 2,048 rows, the ones that reach those kernels, are
compared: there the Gram product's 2^-43 is a fiftieth of the bound."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["random", "graded"])
@pytest.mark.parametrize("name", ["hub15", "spin30"])
def test_against_lapack(name, kind):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    ctx = ed.build_sectors(W.hubbard_chain(15, 1.0, 4.0, 7, 8) if name == "hub15" else
                           W.j1j2_torus(6, 5, 1.0, 0.5, 12, cut_mask=0x7FFF))
    _, dA, dB, _ = ctx.blocks()
    g = torch.Generator(device="cuda")
    g.manual_seed(15)
    x = torch.randn(ctx.dim, device="cuda", dtype=torch.float64, generator=g)
    off = np.concatenate([[0], np.cumsum(dA * dB)])
    blocks = [x[off[i]:off[i + 1]].view(int(dA[i]), int(dB[i])) for i in range(len(dA))]
    if kind == "graded":
        for b in blocks:
            b.mul_(torch.logspace(0, -3, b.shape[0], device="cuda", dtype=torch.float64)[:, None])
    x /= torch.linalg.vector_norm(x)
    es = ed.entanglement_spectrum(ctx, x)
    for b, lam in zip(blocks, es.lam):
        m = min(b.shape)
        if m <= 2048:
            continue
        G = b @ b.T if b.shape[0] <= b.shape[1] else b.T @ b
        ref = torch.linalg.eigvalsh(G).flip(0).cpu().numpy()
        assert np.abs(lam - ref).max() <= m * 2.0 ** -48 * ref[0]
