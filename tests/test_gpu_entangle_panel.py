"""The one-launch panel reduction of the entanglement spectrum at its edges:
Gram matrices of one row, of less than a panel, of a panel's edge (55, 66 and
70 rows: one CTA, then three), of ragged row chunks (286, 495, 1287 and 1716
rows, odd and even), in both orientations of the block.  States: random; of
rank 3 (almost every column of the reduction vanishes); and with rows graded
over 12 decades.  Against the squared singular values of the block from LAPACK
in FP64, to 1e-12 absolute for a normalised state: the reduction's backward
error is about sqrt(m) units of 2^-48 of the largest eigenvalue (<= 1), 1.5e-13
at m = 1716."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["random", "rank3", "graded"])
@pytest.mark.parametrize("L,n_up,n_dw", [(5, 5, 2), (6, 3, 2), (11, 2, 2), (12, 2, 2), (8, 4, 4), (13, 3, 2),
                                         (13, 3, 4), (12, 4, 5), (13, 5, 5), (13, 6, 6)])
def test_panel_reduction_edges(L, n_up, n_dw, kind):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    ctx = ed.build_sectors(W.hubbard_chain(L, 1.0, 4.0, n_up, n_dw))
    _, dA, dB, _ = ctx.blocks()
    dA, dB = int(dA[0]), int(dB[0])
    assert dA * dB == ctx.dim
    rng = np.random.default_rng(dA + 7 * dB)
    if kind == "rank3":
        psi = rng.standard_normal((dA, 3)) @ rng.standard_normal((3, dB))
    else:
        psi = rng.standard_normal((dA, dB))
        if kind == "graded":
            psi *= np.logspace(0, -12, dA)[:, None]
    psi /= np.linalg.norm(psi)
    ref = np.linalg.svd(psi, compute_uv=False) ** 2
    es = ed.entanglement_spectrum(ctx, torch.tensor(psi.ravel(), device="cuda"))
    assert es.lam[0].shape == ref.shape
    assert np.abs(es.lam[0] - ref).max() <= 1e-12
