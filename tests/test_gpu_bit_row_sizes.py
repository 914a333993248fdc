"""Bit rows where a warp writes several chunks (n times chunks from 400,000 on), about
the 16,384 transactions of a chunk with many items, and supports above 2^24."""
import os

import numpy as np
import pytest

import datagen
import oracle

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


def _short_lists(m, n, longest, seed):
    """Lists of 0 to `longest` tids, some at the ends of [0, m), a few long ones among them."""
    rng = np.random.default_rng(seed)
    lists = []
    for i in range(n):
        k = int(rng.integers(0, longest + 1)) if i % 2_000 else min(m, 5_000)
        x = np.unique(rng.integers(0, m, k))
        if i % 5 == 0:
            x = np.unique(np.concatenate([x, [0, m - 1]]))
        lists.append(x.astype(np.uint32))
    lists[0], lists[-1] = np.zeros(0, np.uint32), np.zeros(0, np.uint32)
    return datagen.from_lists(lists, m)


def _sampled(inst, full, seed):
    import torch
    rng = np.random.default_rng(seed)
    n = inst.n
    long_ = np.arange(0, n, 2_000)[1:]
    si = np.concatenate([rng.integers(0, n - 1, 20_000), np.repeat(long_, 200)])
    sj = np.concatenate([rng.integers(0, n, 20_000), rng.integers(0, n, long_.size * 200)])
    keep = si != sj
    ii, jj = np.minimum(si, sj)[keep], np.maximum(si, sj)[keep]
    got = full[torch.from_numpy(oracle.packed_index(n, ii, jj)).cuda()].cpu().numpy().astype(np.uint32)
    assert np.array_equal(got, oracle.pairs_list(inst.offsets, inst.tids, ii, jj, threads=THREADS))


@pytest.mark.parametrize("m,n", [(16_383, 10_000), (16_384, 10_000), (16_385, 10_000), (170_001, 40_000)])
@pytest.mark.parametrize("shuffled", [False, True])
def test_many_items(m, n, shuffled):
    import torch
    import paper_1102_1003_gb300 as pkg
    inst = _short_lists(m, n, 60, seed=m)
    rng = np.random.default_rng(1)
    lists = [inst.tidlist(i) for i in range(n)]
    if shuffled:  # the dense call takes lists in any order
        lists = [rng.permutation(x) if i % 3 == 0 else x for i, x in enumerate(lists)]
    off = torch.from_numpy(inst.offsets.astype(np.int64)).cuda()
    tids = torch.from_numpy(np.concatenate(lists).astype(np.int32)).cuda()
    full = torch.full((n * (n - 1) // 2,), -1, dtype=torch.int32, device="cuda")
    pkg.pair_support_dense(m, off, tids, 2**32 - 1, pairs=torch.empty((1, 3), dtype=torch.int32, device="cuda"), full=full)
    assert int(full.min()) >= 0
    _sampled(inst, full, m)
    del full
    pkg.batmap_release_scratch()
    torch.cuda.empty_cache()


def test_many_items_row_major():
    """The rows of k-way sets, refused where a list is out of order."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m, n = 170_001, 40_000
    inst = _short_lists(m, n, 60, seed=9)
    off = torch.from_numpy(inst.offsets.astype(np.int64)).cuda()
    tids = torch.from_numpy(inst.tids.astype(np.int32)).cuda()
    b = pkg.batmap_build_d(3, m, off, tids)
    rng = np.random.default_rng(2)
    long_ = np.arange(0, n, 2_000)[1:]
    qs = np.stack([rng.choice(long_, 3_000), rng.integers(0, n, 3_000), rng.choice(long_, 3_000)], 1).astype(np.int32)
    for k in (1, 2, 3):
        q = np.ascontiguousarray(qs[:, :k])
        got = pkg.itemset_support(b, torch.from_numpy(q).cuda()).cpu().numpy().astype(np.uint64)
        assert np.array_equal(got, oracle.kway_counts(inst.offsets, inst.tids, q.tolist()))
    b.free()
    e = int(inst.offsets[4_000])  # a long list: tids 4,095 and 4,096 change places
    tids[[e + 4_095, e + 4_096]] = tids[[e + 4_096, e + 4_095]]
    with pytest.raises(pkg.BatmapError) as err:
        pkg.batmap_build_d(3, m, off, tids)
    assert err.value.code == pkg.BATMAP_ERR_ARG


def test_supports_above_2_24():
    """K is split so that a unit spans at most 2^24 transactions; larger supports come from the
    added pieces.  Three lists of every transaction, one of all but a few, and short ones."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m, n = (1 << 24) + (1 << 23) + 77, 1_000
    rng = np.random.default_rng(3)
    short = [np.unique(rng.integers(0, m, 300)) for _ in range(n - 4)]
    gone = np.unique(rng.integers(0, m, 1_000))
    every = torch.arange(m, dtype=torch.int32, device="cuda")
    most = every[~torch.isin(every, torch.from_numpy(gone).cuda().int())]
    lists = [every, most] + [torch.from_numpy(x.astype(np.int32)).cuda() for x in short] + [every, every]
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(torch.tensor([x.numel() for x in lists], device="cuda"), 0)
    b = pkg.batmap_build(m, off, torch.cat(lists))
    full = torch.full((n * (n - 1) // 2,), -1, dtype=torch.int32, device="cuda")
    pkg.pair_support_all(b, 2**32 - 1, pairs=torch.empty((1, 3), dtype=torch.int32, device="cuda"), full=full)
    assert pkg.batmap_get_timing(b)["scan_ms"] == 0  # by the bit rows
    got = full.cpu().numpy().astype(np.int64)
    at = lambda i, j: got[int(oracle.packed_index(n, np.array([min(i, j)]), np.array([max(i, j)]))[0])]
    assert [at(0, 1), at(0, n - 2), at(0, n - 1), at(n - 2, n - 1), at(1, n - 1)] == [m - gone.size, m, m, m, m - gone.size]
    for i, x in enumerate(short[:200]):
        assert at(0, i + 2) == at(n - 1, i + 2) == x.size
        assert at(1, i + 2) == np.setdiff1d(x, gone).size
    for i, j in rng.integers(0, n - 4, (2_000, 2)):
        if i != j:
            assert at(i + 2, j + 2) == np.intersect1d(short[i], short[j]).size
    b.free()
    pkg.batmap_release_scratch()
    torch.cuda.empty_cache()
