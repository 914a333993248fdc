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


@pytest.mark.parametrize("na,nb", [(1, 1), (1, 241), (127, 240), (129, 239), (256, 241), (257, 480), (300, 7)])
def test_cross_tile_edges(na, nb):
    """Cross mode: rows end with family A inside a tile, columns start at family B."""
    import torch
    import paper_1102_1003_gb300 as pkg
    inst = datagen.zipf_tidlists(20_011, na + nb, 0.05, seed=na * 1000 + nb)
    off, tids, _ = device_inputs(inst, 0)
    ref = oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS)
    a, b = np.meshgrid(np.arange(na), np.arange(nb), indexing="ij")
    want = ref[oracle.packed_index(inst.n, a.ravel(), na + b.ravel())]
    for probe_log in (0, 2):  # the library's choice, and a BatMap route
        s = pkg.batmap_build_cross(inst.m, na, off, tids, params=pkg.batmap_default_params(probe_log=probe_log))
        full = torch.full((na * nb,), -1, dtype=torch.int32, device="cuda")
        pkg.pair_support_all(s, 1, full=full)
        assert np.array_equal(full.cpu().numpy().astype(np.uint32), want), probe_log


def test_batch_of_both_routes():
    """One batched pass over sets on either route, small and large, split and whole K."""
    import torch
    import paper_1102_1003_gb300 as pkg
    insts = [datagen.zipf_tidlists(150_000, 700, 0.02, seed=1, s=150), datagen.bernoulli_tidlists(900, 33, 0.2, seed=2, s=3),
             datagen.zipf_tidlists(40_000, 250, 0.04, seed=3, s=40), datagen.bernoulli_tidlists(300, 2, 0.5, seed=4, s=1)]
    sets, fulls, bufs, refs = [], [], [], []
    for q, inst in enumerate(insts):
        off, tids, _ = device_inputs(inst, 0)
        p = pkg.batmap_default_params(probe_log=2) if q == 2 else None
        sets.append(pkg.batmap_build(inst.m, off, tids, params=p))
        refs.append(oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS))
        fulls.append(torch.full((refs[-1].size,), -1, dtype=torch.int32, device="cuda"))
        bufs.append(torch.empty((refs[-1].size, 3), dtype=torch.int32, device="cuda"))
    for rep in range(2):
        n_out = pkg.pair_support_batch(sets, [i.s for i in insts], bufs, fulls)
        for q, inst in enumerate(insts):
            assert np.array_equal(fulls[q].cpu().numpy().astype(np.uint32), refs[q]), (rep, q)
            want = oracle.threshold_from_full(refs[q], inst.n, inst.s)
            assert n_out[q] == want.shape[0]
            assert np.array_equal(bufs[q][:n_out[q]].cpu().numpy().astype(np.uint32), want)
            fulls[q].fill_(-1)


def test_invalid_lists_refused_with_bit_rows():
    """The bit rows' build stands in for the list check: the same lists are refused."""
    import torch
    import paper_1102_1003_gb300 as pkg
    inst = datagen.bernoulli_tidlists(70_000, 50, 0.1, seed=8)
    off, tids, _ = device_inputs(inst, 0)
    e = int(inst.offsets[7]) + 4_000  # inside item 7
    for at, value in ((e, int(inst.tids[e + 1])), (e, 70_000), (e, 0), (int(inst.offsets[50]) - 1, 1 << 30)):
        bad = tids.clone()
        bad[at] = value
        with pytest.raises(pkg.BatmapError) as err:
            pkg.batmap_build(inst.m, off, bad)
        assert err.value.code == pkg.BATMAP_ERR_ARG
    pkg.batmap_build(inst.m, off, tids)


@pytest.mark.parametrize("d", [3, 4])
@pytest.mark.parametrize("m", [200, 8_191, 8_193, 40_007])
def test_kway_supports_of_bit_rows_and_batmaps(d, m):
    """k_bits_support (few and many queries, runs of queries sharing all ids but the last
    that start and end inside its groups) and the BatMap kernels give the merge counts."""
    import torch
    import paper_1102_1003_gb300 as pkg
    inst = datagen.zipf_tidlists(m, 60, 0.1, seed=m + d)
    off, tids, _ = device_inputs(inst, 0)
    sets = [pkg.batmap_build_d(d, m, off, tids, params=pkg.batmap_default_params(probe_log=pl)) for pl in (0, 3)]
    rng = np.random.default_rng(m)
    for k in range(1, d + 1):
        few = rng.integers(0, inst.n, (37, k))
        runs = [np.concatenate([np.tile(rng.integers(0, inst.n, (1, k - 1)), (r, 1)),
                                rng.integers(0, inst.n, (r, 1))], axis=1) for r in rng.integers(1, 21, 260)]
        for qs in (few, np.concatenate(runs)):
            qs = np.ascontiguousarray(qs, np.int32)
            want = oracle.kway_counts(inst.offsets, inst.tids, qs.tolist())
            for s in sets:
                got = pkg.itemset_support(s, torch.from_numpy(qs).cuda()).cpu().numpy().astype(np.uint64)
                assert np.array_equal(got, want), (k, qs.shape)


@pytest.mark.parametrize("d", [3, 4])
def test_frequent_itemsets_same_on_both_routes(d):
    """Triples (and quadruples) of a set with bit rows equal those of the BatMap kernels."""
    import paper_1102_1003_gb300 as pkg
    inst = datagen.zipf_tidlists(30_000, 200, 0.04, seed=9)
    off, tids, _ = device_inputs(inst, 0)
    s = 40
    b2 = pkg.batmap_build(inst.m, off, tids)
    _, pairs = pkg.pair_support_all(b2, s)
    got = []
    for pl in (0, 3):
        b = pkg.batmap_build_d(d, inst.m, off, tids, params=pkg.batmap_default_params(probe_log=pl))
        n3, t3, c3 = pkg.frequent_triples(b, s, pairs)
        r = [n3, c3, t3.cpu().numpy()]
        if d == 4:
            n4, t4, c4 = pkg.frequent_quadruples(b, s, t3)
            r += [n4, c4, t4.cpu().numpy()]
        got.append(r)
    assert got[0][0] > 0
    for x, y in zip(*got):
        assert np.array_equal(x, y)
