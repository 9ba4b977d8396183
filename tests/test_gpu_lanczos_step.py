"""The Lanczos step in one launch, in a cluster of 8 or 16 CTAs (1 to 32,768
states; here 1, 2, 462, 4,900, 10,584, 12,870 and 30,240) and in a cooperative grid
(from 131,072; here 213,444 and 853,776), and the three launches between
(44,100), in FP64 with the exact fixed-point H|psi>, with couplings that are not
dyadic, and with FP32 vectors.
The first 12 alpha, beta against the same recurrence in FP64 on the host with the
oracle's H|psi>: 1e-11 of the largest in FP64 (12 steps of rounding, no
re-orthogonalisation yet needed), 2e-5 in FP32; two runs give the same bits."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def _models():
    return {"one": W.hubbard_chain(3, 1.0, 4.0, 3, 3), "two": W.heisenberg_chain(2, cut_mask=1),
            "hub8": W.hubbard_chain(8, 1.0, 4.0, 4, 4), "xxz11": W.xxz_chain(11, 1.0, 0.5, n_up=5, cut_mask=0x1F),
            "heis16": W.config_heis16(), "j03": W.j1j2_torus(4, 4, 1.0, 0.3, cut_mask=0xFF),
            "hub9": W.hubbard_chain(9, 1.0, 4.0, 3, 5, tp=0.3), "hub10": W.hubbard_chain(10, 1.0, 4.0, 3, 5),
            "three": W.hubbard_chain(10, 1.0, 4.0, 4, 4), "hub11": W.hubbard_chain(11, 1.0, 4.0, 5, 5),
            "hub12": W.config_hub12()}


@pytest.mark.parametrize("name", ["one", "two", "hub8", "xxz11", "hub9", "heis16", "j03", "hub10", "three",
                                  "hub11", "hub12"])
def test_recurrence(oracle_mod, name):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    m = _models()[name]
    ctx = ed.build_local_ops(ed.build_sectors(m))
    keys, okeys = ctx.state_keys(), oracle_mod.sector_keys(m)
    v = W.start_values(okeys)
    v = v / np.linalg.norm(v)
    x = torch.tensor(v[oracle_mod.find_keys(m, okeys, keys)], device="cuda")
    steps = min(12, max(1, len(okeys) - 1))
    a, b, vp, bt = [], [], np.zeros_like(v), 0.0
    for _ in range(steps):
        w = oracle_mod.apply_H(m, okeys, v) - bt * vp
        a.append(v @ w)
        w = w - a[-1] * v
        bt = np.linalg.norm(w)
        b.append(bt)
        vp, v = v, w / (bt if bt > 0 else 1.0)
    scale = np.abs(a).max() + np.abs(b).max()
    for mode, tol in (("f64", 1e-11), ("f32", 2e-5)):
        r, s = (ed.lanczos_ground(ctx, mode, max_iter=steps + 2, fixed_iter=True, v0=x) for _ in range(2))
        k = min(steps, len(r.alpha))
        assert np.abs(r.alpha[:k] - a[:k]).max() <= tol * scale
        assert np.abs(r.beta[:k] - b[:k])[: max(1, k - 1)].max() <= tol * scale
        assert np.array_equal(r.alpha, s.alpha) and np.array_equal(r.beta, s.beta)
