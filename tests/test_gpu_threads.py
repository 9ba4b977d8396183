"""Host threads with a context and a stream each.  H|psi> of eight contexts whose
widest rows differ but share a kernel instantiation (3,432 and 6,435 columns: two
CTAs of the row pass per SM; the same on the general path), 5,000 times each at
once; every result has the bits of the context alone."""
import threading

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


def _at_once(jobs):
    import torch

    errors, gate = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            torch.cuda.set_device(0)
            s = torch.cuda.Stream()
            gate.wait()
            with torch.cuda.stream(s):
                job()
            s.synchronize()
        except BaseException as e:  # reported by the test's thread
            errors.append(e)

    th = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in th:
        t.start()
    for t in th:
        t.join()
    assert not errors, errors


def _chain(nA, nB, n_up, spread):
    n = nA + nB
    J = 1.0 + (np.arange(n) * 0.37 % 1.0 if spread else np.zeros(n))  # spread: more than four value classes
    return W.Model("spin", n, W.chain_bonds(n, True), jxy=list(J), jz=list(J), n_up=n_up, cut_mask=(1 << nA) - 1)


@pytest.mark.parametrize("path", ["k_row5", "general"])
def test_apply_contexts_of_different_width(ed, path):
    import torch

    ctxs = [ed.build_local_ops(ed.build_sectors(_chain(1, nB, k, path == "general"))) for nB, k in ((14, 7), (15, 7)) * 4]
    assert [int(max(c.blocks()[2])) for c in ctxs] == [3432, 6435] * 4
    assert all((c.row_pass(torch.float64) == "k_row5") == (path == "k_row5") for c in ctxs)
    xs = [torch.randn(c.dim, device="cuda", dtype=torch.float64) for c in ctxs]
    refs = [ed.apply_H(c, x, torch.empty_like(x)).clone() for c, x in zip(ctxs, xs)]
    outs = [[torch.empty_like(x) for _ in range(3)] for x in xs]
    torch.cuda.synchronize()

    def job(c, x, out):
        def run():
            for i in range(5000):
                ed.apply_H(c, x, out[i % 3])
        return run

    _at_once([job(*a) for a in zip(ctxs, xs, outs)])
    assert all(torch.equal(o, r) for out, r in zip(outs, refs) for o in out)
