"""The bit-row contraction at the edges of its tiles (256 rows x 240 columns,
K blocks of 256, chunks of 32,768 transactions), against the merge oracle.
Every comparison is exact: supports are integers."""
import os

import numpy as np
import pytest

import datagen
import oracle
from tests.gpu_util import device_inputs

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)


def _dense_full(inst, tids=None):
    import torch
    import paper_1102_1003_gb300 as pkg
    off, t, _ = device_inputs(inst, 0)
    npairs = inst.n * (inst.n - 1) // 2
    full = torch.full((max(npairs, 1),), -1, dtype=torch.int32, device="cuda")
    pkg.pair_support_dense(inst.m, off, t if tids is None else tids, 1, full=full)
    return full[:npairs].cpu().numpy().astype(np.uint32)


@pytest.mark.parametrize("n", [2, 127, 128, 129, 239, 240, 241, 256, 257, 480, 481, 513])
def test_tile_edges(n):
    inst = datagen.bernoulli_tidlists(2_049, n, 0.1, seed=n)
    assert np.array_equal(_dense_full(inst), oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS))


@pytest.mark.parametrize("m", [1, 255, 256, 257, 511, 1_025, 32_767, 32_768, 32_769, 65_537])
def test_block_and_chunk_edges(m):
    inst = datagen.bernoulli_tidlists(m, 70, 0.3, seed=m)
    assert np.array_equal(_dense_full(inst), oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS))


def test_unsorted_lists():
    """pair_support_dense takes the lists in any order."""
    import torch
    inst = datagen.zipf_tidlists(100_001, 60, 0.05, seed=5)
    rng = np.random.default_rng(6)
    shuffled = np.concatenate([rng.permutation(inst.tidlist(i)) for i in range(inst.n)])
    got = _dense_full(inst, torch.from_numpy(shuffled.astype(np.int32)).cuda())
    assert np.array_equal(got, oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS))


def test_largest_supports():
    """m = 2^24, the limit of exact FP32 partial sums: full and nearly full rows."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m = 1 << 24
    rows = [np.arange(m), np.arange(m - 1), np.arange(1, m, 2), np.arange(0, m, 3), np.arange(m)]
    member = np.zeros((5, m), bool)
    for i, r in enumerate(rows):
        member[i, r] = True
    want = [int((member[i] & member[j]).sum()) for i in range(5) for j in range(i + 1, 5)]
    off = torch.from_numpy(np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int64)).cuda()
    tids = torch.from_numpy(np.concatenate(rows).astype(np.int32)).cuda()
    full = torch.zeros(10, dtype=torch.int32, device="cuda")
    pkg.pair_support_dense(m, off, tids, 1, full=full)
    assert full.tolist() == want
