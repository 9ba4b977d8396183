"""The launches of one batched H|psi> follow one another where they overlap: a
batch with CSR, 64-wide and 128-wide instances at once, applied to six different
vectors back to back on one stream (a product that started before the pieces of
its own vector were complete would mix two of them), gives the bits of the same
applies with the GPU idle in between."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_back_to_back_applies():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    ms = [W.hubbard_chain(L, 1.0, 3.0, u, d, tp=0.2)
          for L, u, d in [(13, 6, 1), (12, 6, 6), (9, 4, 1), (12, 5, 4), (10, 5, 2), (8, 1, 2), (12, 6, 1)]]
    b = ed.batch_create(ms, flags=2)
    assert set(np.asarray(b.info()[0]).tolist()) == {0, 1, 2}
    g = torch.Generator(device="cuda")
    g.manual_seed(11)
    xs = [torch.randn(b.dim, device="cuda", dtype=torch.float32, generator=g) for _ in range(6)]
    ys, zs = ([torch.full_like(x, float("nan")) for x in xs] for _ in range(2))
    for x, z in zip(xs, zs):
        ed.batch_apply(b, x, z)
        torch.cuda.synchronize()
    for _ in range(5):
        for y in ys:
            y.fill_(float("nan"))
        for x, y in zip(xs, ys):
            ed.batch_apply(b, x, y)
        torch.cuda.synchronize()
        assert all(torch.equal(y, z) for y, z in zip(ys, zs))
