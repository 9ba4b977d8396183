"""H|psi> with column counts on both sides of the row pass's 32-column slabs and of
the panel pass's 128 (FP64) and 256 columns (FP32), the side dimensions nearest to
those edges: 30 and 35, 126 and 136, 253 and 276 (31 to 33, 127 to 129 and 255 to
257 columns need a side of more than the 30 sites that one may have).  Without
cross terms (Hubbard; several rows per side A state) and with them (spin, two
sites against the rest).  Against the oracle, FP64 and FP32; tolerances as in
test_gpu_apply (relative L2 1e-12 / 1e-6)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

HUB = {30: (30, 1), 35: (7, 3), 36: (9, 2), 120: (10, 3), 126: (9, 4), 136: (17, 2),
       253: (23, 2), 276: (24, 2)}
SPIN = {30: (30, 1), 35: (7, 3), 36: (9, 2), 120: (16, 2), 126: (9, 4), 136: (17, 2), 253: (23, 2), 276: (24, 2)}


@pytest.mark.parametrize("kind,dB", [("hub", d) for d in HUB] + [("spin", d) for d in SPIN])
def test_column_edges(oracle_mod, kind, dB):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    if kind == "hub":
        n, k = HUB[dB]
        m = W.hubbard_chain(n, 1.0, 4.0, 1, k)
    else:
        n, k = SPIN[dB]
        m = W.heisenberg_chain(n + 2, n_up=k, pbc=True, cut_mask=3)
    ctx = ed.build_local_ops(ed.build_sectors(m))
    assert dB in [int(d) for d in ctx.blocks()[2]]
    assert ctx.row_pass(torch.float64) == "k_row5" and ctx.row_pass(torch.float32) == "k_row5"
    keys, okeys = ctx.state_keys(), oracle_mod.sector_keys(m)
    pos = oracle_mod.find_keys(m, okeys, keys)
    y_ref = oracle_mod.apply_H(m, okeys, W.start_values(okeys))[pos]
    for dt, tol in ((torch.float64, 1e-12), (torch.float32, 1e-6)):
        x = torch.tensor(W.start_values(keys), device="cuda").to(dt)
        y = torch.full_like(x, float("nan"))
        ed.apply_H(ctx, x, y)
        err = np.linalg.norm(y.double().cpu().numpy() - y_ref) / np.linalg.norm(y_ref)
        assert err <= tol, (dt, err)
