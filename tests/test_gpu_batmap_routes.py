"""The routes that a set without bit rows takes (tile, shape_mask or probe_log set, or
no memory for the rows): cyclic scan and probe of pairs, their corrections, the witness
scans and probes of triples and quadruples.  Every comparison is exact."""
import os

import numpy as np
import pytest

import datagen
import oracle
from oracle import dof_rules as R
from tests.gpu_util import device_inputs, run_all_pairs

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


def _corrections(inst, bset):
    """Number of (failed tid, pair holding it) from the exported failure lists."""
    import paper_1102_1003_gb300 as pkg
    failed = np.bincount(pkg.batmap_export_layout(bset)["fail_tids"], minlength=inst.m).astype(np.int64)
    holders = np.bincount(inst.tids, minlength=inst.m).astype(np.int64)
    return int((failed * (holders - 1) - failed * (failed - 1) // 2).sum())


FORCED = [dict(max_loop=1), dict(load_num=1, load_den=1), dict(load_num=1, load_den=2, max_loop=2),
          dict(load_num=1, load_den=8, max_loop=1)]


@pytest.mark.parametrize("probe_log", [0, 2, 32])  # bit rows; scan and probe; scan alone
@pytest.mark.parametrize("params", FORCED)
def test_forced_failures(params, probe_log):
    import paper_1102_1003_gb300 as pkg
    rng = np.random.default_rng(5)
    zipf = datagen.zipf_tidlists(20_000, 120, 0.08, seed=11, s=20)
    full_item = datagen.from_lists([np.arange(5_000, dtype=np.uint32)] +
                                   [np.flatnonzero(rng.random(5_000) < 0.3).astype(np.uint32) for _ in range(9)], 5_000, s=1)
    for inst in (zipf, full_item):
        full, n_out, pairs, b = run_all_pairs(inst, perm_seed=3, params=pkg.batmap_default_params(probe_log=probe_log, **params))
        ref = oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS)
        assert np.array_equal(full, ref)
        assert np.array_equal(pairs, oracle.threshold_from_full(ref, inst.n, inst.s))
        info = b.info
        assert info["n_corrections"] == _corrections(inst, b)
        # (the full item's family takes load 1 without a failure)
        assert info["n_failed"] > 0 or (inst is full_item and params.get("load_den") == 1)
        assert (pkg.batmap_get_timing(b)["scan_ms"] > 0) == (probe_log > 0)


@pytest.mark.parametrize("probe_log", [2, 32])
@pytest.mark.parametrize("na,nb", [(150, 220), (1, 300), (257, 3)])
def test_cross_forced_failures(na, nb, probe_log):
    import torch
    import paper_1102_1003_gb300 as pkg
    a, b = datagen.zipf_tidlists(40_000, na, 0.03, seed=na), datagen.bernoulli_tidlists(40_000, nb, 0.02, seed=nb)
    u = datagen.from_lists([a.tidlist(i) for i in range(na)] + [b.tidlist(j) for j in range(nb)], 40_000)
    off, tids, _ = device_inputs(u, 5)
    s = pkg.batmap_build_cross(u.m, na, off, tids, params=pkg.batmap_default_params(
        max_loop=1, load_num=1, load_den=2, probe_log=probe_log))
    assert s.info["n_failed"] > 0 and s.info["n_corrections"] == _corrections(u, s) > 0
    full = torch.full((na * nb,), -1, dtype=torch.int32, device="cuda")
    pkg.pair_support_all(s, 1, full=full)
    assert pkg.batmap_get_timing(s)["scan_ms"] > 0
    i, j = np.meshgrid(np.arange(na), np.arange(nb), indexing="ij")
    ref = oracle.pairs_full(u.offsets, u.tids, threads=THREADS)[oracle.packed_index(u.n, i.ravel(), na + j.ravel())]
    assert np.array_equal(full.cpu().numpy().astype(np.uint32), ref)


def _levels(inst, s, depth):
    """Candidates and frequent itemsets of sizes 3 to `depth` by merges."""
    pairs = oracle.pairs_threshold(inst.offsets, inst.tids, s)
    out, below = [], pairs[:, :2]
    for k in range(3, depth + 1):
        cand = R.triple_candidates(below) if k == 3 else R.quadruple_candidates(below)
        sup = oracle.kway_counts(inst.offsets, inst.tids, cand.tolist())
        hits = np.concatenate([cand[sup >= s], sup[sup >= s, None].astype(np.uint32)], axis=1).astype(np.uint32)
        out.append((cand, hits))
        below = hits[:, :k]
    return pairs, out


@pytest.mark.parametrize("params", [{}, dict(max_loop=1, load_num=1, load_den=1), dict(max_loop=1, load_num=1, load_den=2)])
@pytest.mark.parametrize("d", [3, 4])
def test_itemset_scans_and_probes(d, params):
    """Items of three densities, so that candidates go to the scan (similar widths) and to the probe
    (the widest 8 times the narrowest, 2 times for d = 4)."""
    import torch
    import paper_1102_1003_gb300 as pkg
    rng = np.random.default_rng(17 + d)
    m, counts = (20_000, (10, 20, 30)) if d == 3 else (12_000, (6, 8, 10))
    lists = [np.flatnonzero(rng.random(m) < p).astype(np.uint32)
             for p, c in zip((0.5, 0.12, 0.03) if d == 3 else (0.6, 0.15, 0.04), counts) for _ in range(c)]
    inst = datagen.from_lists(lists, m, s=1)
    ref_pairs, levels = _levels(inst, 1, d)
    off, tids, _ = device_inputs(inst, 7)
    pairs = torch.from_numpy(ref_pairs.astype(np.int32)).cuda()
    b = pkg.batmap_build_d(d, m, off, tids, params=pkg.batmap_default_params(probe_log=3, perm_seed=7, **params))
    if params:
        assert b.info["n_failed"] > 0
    below = pairs
    for cand, hits in levels:
        call = pkg.frequent_triples if cand.shape[1] == 3 else pkg.frequent_quadruples
        n_out, got, n_cand = call(b, 1, below)
        t = pkg.batmap_get_timing(b)
        assert t["scan_ms"] > 0 and t["probe_ms"] > 0
        assert n_cand == cand.shape[0] and n_out == hits.shape[0]
        assert np.array_equal(got.cpu().numpy().astype(np.uint32), hits)
        below = got


@pytest.mark.parametrize("d", [3, 4])
def test_item_failing_almost_entirely(d):
    """Load 1/4 per slot and one round of moves: most elements of the wide items are found by the
    failure lists alone."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m = 20_000
    inst = datagen.from_lists([np.arange(a, m, b, dtype=np.uint32) for a, b in ((0, 2), (0, 3), (0, 5), (1, 7), (0, 4))], m)
    off, tids, _ = device_inputs(inst, 2)
    b = pkg.batmap_build_d(d, m, off, tids, params=pkg.batmap_default_params(load_num=1, load_den=4, max_loop=1, probe_log=3))
    assert b.info["n_failed"] > 1_000
    for k in range(1, d + 1):
        qs = np.random.default_rng(k).integers(0, 5, (400, k)).astype(np.int32)
        got = pkg.itemset_support(b, torch.from_numpy(qs).cuda()).cpu().numpy().astype(np.uint64)
        assert np.array_equal(got, oracle.kway_counts(inst.offsets, inst.tids, qs.tolist())), k


def test_autotuned_scan_in_a_batch():
    """The tuned schedule is the one that a batch of sets on the scan runs."""
    import torch
    import paper_1102_1003_gb300 as pkg
    insts = [datagen.batch_instance(sp) for sp in datagen.batch_specs(5, 2000, m_range=(1e4, 1e5), n_range=(100, 700))]
    sets = []
    for inst in insts:
        off, tids, _ = device_inputs(inst, 0)
        sets.append(pkg.batmap_build(inst.m, off, tids, params=pkg.batmap_default_params(probe_log=2)))
    eff = pkg.batmap_autotune(sets)
    assert max(eff) == pytest.approx(1.0) and min(eff) > 0
    refs = [oracle.pairs_full(i.offsets, i.tids, threads=THREADS) for i in insts]
    fulls = [torch.full((r.size,), -1, dtype=torch.int32, device="cuda") for r in refs]
    bufs = [torch.empty((max(int((r >= i.s).sum()), 1), 3), dtype=torch.int32, device="cuda") for r, i in zip(refs, insts)]
    n_out = pkg.pair_support_batch(sets, [i.s for i in insts], bufs, fulls)
    for q, inst in enumerate(insts):
        want = oracle.threshold_from_full(refs[q], inst.n, inst.s)
        assert np.array_equal(fulls[q].cpu().numpy().astype(np.uint32), refs[q]) and n_out[q] == want.shape[0]
        assert np.array_equal(bufs[q][:n_out[q]].cpu().numpy().astype(np.uint32), want)
        assert sets[q].info["n_work_units"] > 0
        pkg.pair_support_all(sets[q], inst.s, full=fulls[q])
        assert pkg.batmap_get_timing(sets[q])["scan_ms"] > 0


def _bernoulli_on_device(m, n, p, seed):
    """CSR tidlists made on the device (geometric gaps), for sizes that take minutes on the host."""
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    width = int(m * p + 8 * (m * p) ** 0.5)
    sizes, parts = [], []
    for i in range(0, n, 256):
        gaps = torch.rand((min(256, n - i), width), generator=gen, device="cuda", dtype=torch.float64).clamp_(min=1e-300)
        pos = gaps.log_().div_(np.log1p(-p)).ceil_().clamp_(min=1.0).cumsum_(1).sub_(1.0)
        keep = pos < m
        sizes.append(keep.sum(1))
        parts.append(pos[keep].to(torch.int32))
    off = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.cat(sizes), 0, out=off[1:])
    return off, torch.cat(parts)


def test_scan_at_full_size():
    """m = 2^22, n = 8,192, 5%: the scan over 12.9 GB of BatMaps against the contraction of the bit
    rows, which the full-size tests compare with merges; 64 pairs by merges here."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m, n = 1 << 22, 8_192
    off, tids = _bernoulli_on_device(m, n, 0.05, 3)
    fulls = []
    for probe_log in (0, 32):
        b = pkg.batmap_build(m, off, tids, params=pkg.batmap_default_params(probe_log=probe_log))
        fulls.append(torch.full((n * (n - 1) // 2,), -1, dtype=torch.int32, device="cuda"))
        pkg.pair_support_all(b, 2**32 - 1, pairs=torch.empty((1, 3), dtype=torch.int32, device="cuda"), full=fulls[-1])
        assert (pkg.batmap_get_timing(b)["scan_ms"] > 0) == (probe_log > 0)
        assert b.info["bytes"] == n * 3 << 19
        b.free()
    assert torch.equal(fulls[0], fulls[1])
    h = off.tolist()
    rng = np.random.default_rng(4)
    for _ in range(64):
        i, j = sorted(rng.choice(n, 2, replace=False).tolist())
        x, y = (tids[h[k]:h[k + 1]].cpu().numpy() for k in (i, j))
        at = int(oracle.packed_index(n, np.array([i]), np.array([j]))[0])
        assert int(fulls[1][at]) == np.intersect1d(x, y, assume_unique=True).size
    del off, tids, fulls
    pkg.batmap_release_scratch()
    torch.cuda.empty_cache()
