"""Device memory of a batch in dense form: three FP32 vectors, the CSR rows and the
BF16 pieces of H_A, H_B and Psi per instance (rows padded to 64), with 24 MB for the
batch's own lists and history and for the allocator's granularity."""
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_dense_batch_holds_no_more_than_it_uses():
    import torch

    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_07621_gb300 as ed

    ms = [W.hubbard_chain(12, 1.0, 3.0, 6, 5, tp=0.2)] * 48  # 924 x 792
    dA, dB, kA, kB = 924, 792, 960, 832
    nnz = 2 * 12 * (dA + dB)  # ring and next-nearest neighbours: at most 24 entries a row
    per = 12 * dA * dB + 6 * (dA * kA + dB * kB + dA * kB) + 8 * nnz + 16 * (dA + dB) + 65536
    ed.batch_create(ms[:1], flags=2)  # the library's own fixed memory
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    b = ed.batch_create(ms, flags=2)
    held = free - torch.cuda.mem_get_info()[0]
    x = torch.randn(b.dim, device="cuda", dtype=torch.float32)
    ed.batch_apply(b, x, torch.empty_like(x))
    torch.cuda.synchronize()
    assert held <= 48 * per + (24 << 20), (held, 48 * per)
