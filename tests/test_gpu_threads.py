"""Four host threads with their own contexts and streams run spectra and Lanczos
steps at once, whose kernels wait across their CTAs (one launch per panel; one
launch per step in a cooperative grid, 213,444 states, and in a cluster, 4,900):
every result has the bits of the same calls made alone, and no wait runs out."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_spectra_and_steps_at_once():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    def work():
        torch.cuda.set_device(0)
        s = torch.cuda.Stream()
        out = []
        with torch.cuda.stream(s):
            g = torch.Generator(device="cuda")
            g.manual_seed(7)
            c1, c2, c3 = (ed.build_local_ops(ed.build_sectors(W.hubbard_chain(L, 1.0, 4.0, n, n)))
                          for L, n in ((12, 6), (11, 5), (8, 4)))
            x1, x2, x3 = (torch.randn(c.dim, device="cuda", dtype=torch.float64, generator=g) for c in (c1, c2, c3))
            for x in (x1, x2, x3):
                x /= torch.linalg.vector_norm(x)
            for _ in range(4):
                out.append(ed.entanglement_spectrum(c1, x1).lam[0])
                for c, x in ((c2, x2), (c3, x3)):
                    r = ed.lanczos_ground(c, "f64", max_iter=60, fixed_iter=True, v0=x)
                    out += [r.alpha, r.beta]
        return out

    ref = work()
    res, errors = {}, []

    def run(i):
        try:
            res[i] = work()
        except BaseException as e:  # reported below, by the test's thread
            errors.append(e)

    th = [threading.Thread(target=run, args=(i,)) for i in range(4)]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors, errors
    for i in range(4):
        assert all(np.array_equal(a, b) for a, b in zip(res[i], ref)) and len(res[i]) == len(ref)
