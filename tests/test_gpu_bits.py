"""Bit rows by chunks of 4,096 transactions (few items) and of 16,384 (many), at the
ends of both: pair supports against a float32 product of 0/1 rows, exact below 2^24."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [60, 5_000])
@pytest.mark.parametrize("m", [4_095, 4_096, 4_097, 16_385, 32_767, 32_768, 32_769])
def test_supports_by_chunk(n, m):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_1102_1003_gb300 as pkg
    torch.cuda.set_device(0)
    torch.backends.cuda.matmul.allow_tf32 = False
    gen = torch.Generator(device="cuda").manual_seed(m + n)
    p = torch.rand(n, 1, generator=gen, device="cuda") ** 6  # most lists short
    x = torch.rand(n, m, generator=gen, device="cuda") < p
    x[0], x[1], x[2] = True, False, False
    x[2, [0, m - 1]] = True
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = x.sum(1).cumsum(0)
    tids = x.nonzero()[:, 1].to(torch.int32)
    full = torch.zeros(n * (n - 1) // 2, dtype=torch.int32, device="cuda")
    pkg.pair_support_dense(m, off, tids, 1, full=full)
    f = x.to(torch.float32)
    want = (f @ f.T).to(torch.int32)[tuple(torch.triu_indices(n, n, 1, device="cuda"))]
    assert torch.equal(full, want)
    b = pkg.batmap_build(m, off, tids)
    full.zero_()
    pkg.pair_support_all(b, 1, full=full)
    assert torch.equal(full, want)
    b.free()
