"""Dense batched H|psi> at the edges of its tiles: blocks of one row or column,
just below and above 64 and 128, and long thin ones in both orientations (the
64-wide and the 128-wide output tiles, one to fifteen K steps of either
product), alone and all in one batch, with next-nearest-neighbour hopping and
site energies that fill all three BF16 pieces.  Against the oracle in FP64:
1e-6 relative, as for every FP32-storage apply (24 significant bits of every
operand, FP32 sums); twice in a row, and alone or in the batch, the same bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(2, 1, 1), (5, 5, 2), (5, 2, 0), (8, 4, 1), (8, 1, 4), (9, 4, 2), (9, 4, 4), (10, 5, 4), (11, 5, 1),
          (12, 2, 6), (12, 6, 2), (12, 5, 5)]


@pytest.mark.parametrize("flags", [0, 2])
def test_tile_edges(oracle_mod, flags):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    ms = [W.hubbard_chain(L, 1.0, 3.7, u, d, tp=0.2371, eps=np.linspace(-0.813, 0.659, L)) for L, u, d in SHAPES]

    def apply(models, xs):
        b = ed.batch_create(models, flags=flags)
        x = torch.tensor(np.concatenate(xs), dtype=torch.float32, device="cuda")
        y, z = torch.full_like(x, 7.0), torch.full_like(x, -7.0)
        ed.batch_apply(b, x, y)
        ed.batch_apply(b, x, z)
        assert torch.equal(y, z)
        off = b.offsets()
        y = y.double().cpu().numpy()
        return [y[off[i]:off[i + 1]] for i in range(len(models))], b.info()[0]

    xs, refs = [], []
    for m in ms:
        keys, okeys = ed.build_sectors(m).state_keys(), oracle_mod.sector_keys(m)
        x = np.random.default_rng(len(keys)).standard_normal(len(okeys)).astype(np.float32)
        pos = oracle_mod.find_keys(m, okeys, keys)
        xs.append(x[pos])
        refs.append(oracle_mod.apply_H(m, okeys, x.astype(np.float64))[pos])
    together, modes = apply(ms, xs)
    for m, x, ref, y, mode in zip(ms, xs, refs, together, modes):
        assert np.linalg.norm(y - ref) <= 1e-6 * np.linalg.norm(ref), m.name
        if flags == 2:
            (alone,), (one,) = apply([m], [x])
            assert one == mode and np.array_equal(alone, y), m.name
