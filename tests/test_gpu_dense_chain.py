"""Dense-block H|psi> where one output tile sums a chain of products: inner
dimensions around the 64-wide K steps and above the 2,048-wide exact chunks
(two drains of one product inside a chain), and column slicing around its
256-row runs, with an all-zero column.  Against the oracle's block formula;
tolerance as in test_gpu_dense (relative L2 1e-12)."""
import numpy as np
import pytest

import workloads.dense as WD

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chi,pairs", [([1, 2], 1), ([255, 257, 64], 2), ([31, 512, 33], 1), ([2112, 40], 1)])
def test_dense_chain(chi, pairs):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed
    from oracle.dense import dense_apply

    m = WD.dense_block_operator(chi, n_pairs=pairs, seed=77)
    x = np.random.default_rng(6).standard_normal(m.dim)
    off = m.offsets()
    if chi[0] > 2:
        x[off[0]:off[1]].reshape(chi[0], chi[0])[:, 5] = 0.0
        x[off[0]:off[1]].reshape(chi[0], chi[0])[:, 7] *= 1e-9
    op = ed.DenseOperator(m)
    xd = torch.tensor(x, device="cuda")
    yd = torch.full_like(xd, float("nan"))
    op.apply(xd, yd)
    y, y_ref = yd.cpu().numpy(), dense_apply(m, x)
    assert np.linalg.norm(y - y_ref) <= 1e-12 * np.linalg.norm(y_ref)
