"""Green's function with the re-orthogonalisation (FP64 dots, FP32-plane updates), on
shifted sectors of ragged size (16, 100, 225 and 1,225 states: rows that are no
multiple of the 4, 32 or 128 elements the kernels move at a time), from a
random state.  Against the oracle's FP64 run with full re-orthogonalisation;
tolerance 1e-9 of max |G| at eta = 0.5, as in test_gpu_lanczos for the
well-conditioned G."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,n_up,n_dw,n_iter", [(4, 2, 1, 16), (5, 2, 2, 60), (6, 3, 2, 37), (7, 3, 3, 80)])
@pytest.mark.parametrize("reorth", ["full", "partial"])
def test_gf_ragged_sectors(oracle_mod, L, n_up, n_dw, n_iter, reorth):
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    m = W.hubbard_chain(L, 1.0, 4.0, n_up, n_dw, tp=0.25, eps=np.linspace(-0.7, 0.6, L))
    ctx = ed.build_local_ops(ed.build_sectors(m))
    keys, okeys = ctx.state_keys(), oracle_mod.sector_keys(m)
    psi = np.random.default_rng(L).standard_normal(len(okeys))
    psi /= np.linalg.norm(psi)
    omega = np.linspace(-8.0, 8.0, 161)
    ref = oracle_mod.green_function(m, psi, -3.0, omega, 0.5, n_iter=n_iter)
    x = torch.tensor(psi[oracle_mod.find_keys(m, okeys, keys)], device="cuda")
    G, _ = ed.lanczos_gf(ctx, x, -3.0, omega, 0.5, n_iter=n_iter, reorth=reorth)
    assert np.abs(G - ref).max() <= 1e-9 * np.abs(ref).max()
