"""Row pass of H|psi> at the edges of its dispatch: column counts around the
32-column slabs and around the CTA shapes (256, 512 or 1024 threads by the
widest block), cut sites that fill one to four octets of cross-bond slots,
more than two value classes on the cut.  Against the oracle, FP64 and FP32;
tolerances as in test_gpu_apply (relative L2 1e-12 / 1e-6)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _chain(nA, nB, n_up, **kw):
    return W.heisenberg_chain(nA + nB, n_up=n_up, pbc=True, cut_mask=(1 << nA) - 1, **kw)


def _comb(pairs, J, n_up):
    """Side A = sites 0..pairs-1, side B = the rest, one cross bond per pair, and both sides a ring."""
    bonds = W.chain_bonds(pairs, True) + [(i + pairs, j + pairs) for i, j in W.chain_bonds(pairs, True)]
    cross = [(i, i + pairs) for i in range(pairs)]
    return W.Model("spin", 2 * pairs, bonds + cross, jxy=[1.0] * len(bonds) + J, jz=[0.5] * len(bonds) + J, n_up=n_up,
                   cut_mask=(1 << pairs) - 1)


CASES = {
    # widest d_B: 32 +- (31 columns: n_B choose 1), 3432 (512 threads), 6435, 12870 (1024 threads)
    "dB_31": lambda: _chain(2, 31 - 4, 1),
    "dB_20_rows_odd": lambda: _chain(5, 6, 3),
    "dB_3432": lambda: _chain(2, 14, 7),
    "dB_6435": lambda: _chain(3, 15, 7),
    "dB_12870": lambda: _chain(1, 16, 8),
    "hub_dB_3432": lambda: W.hubbard_chain(14, 1.0, 4.0, 1, 7),
    # 9 cross sites: two octets, the second with one entry; two classes
    "comb_9": lambda: _comb(9, [0.5] * 4 + [1.0] * 5, 6),
    # four classes on the cut (chain bonds J = 1 among them): the bond loop
    "comb_6_classes": lambda: _comb(6, [0.5, 0.25, 2.0, 0.5, 0.25, 2.0], 5),
    # every A site bound to every B site: 25 bonds, five on each B site (three
    # entries per site with two classes: 15 to 25 entries, up to four octets)
    "full_5x5": lambda: W.Model("spin", 10, [(i, 5 + j) for i in range(5) for j in range(5)],
                                jxy=[1.0, 0.5, 0.5, 0.5, 1.0] * 5, jz=1.0, n_up=5, cut_mask=31),
}


@pytest.mark.parametrize("name", list(CASES))
def test_row_pass_shapes(oracle_mod, name):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    m = CASES[name]()
    ctx = ed.build_local_ops(ed.build_sectors(m))
    assert ctx.row_pass(torch.float64) == "k_row5" and ctx.row_pass(torch.float32) == "k_row5"
    keys, okeys = ctx.state_keys(), oracle_mod.sector_keys(m)
    pos = oracle_mod.find_keys(m, okeys, keys)
    y_ref = oracle_mod.apply_H(m, okeys, W.start_values(okeys))[pos]
    for dt, tol in ((torch.float64, 1e-12), (torch.float32, 1e-6)):
        x = torch.tensor(W.start_values(keys), device="cuda").to(dt)
        y = torch.full_like(x, float("nan"))
        ed.apply_H(ctx, x, y)
        err = np.linalg.norm(y.double().cpu().numpy() - y_ref) / np.linalg.norm(y_ref)
        assert err <= tol, (name, dt, err)
