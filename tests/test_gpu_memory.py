"""What the library does where device memory runs short (a test limit stands for
the device's size; results are exact all along)."""
import gc
import os

import numpy as np
import pytest

import datagen
import oracle
from tests.gpu_util import device_inputs

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4
MB = 1 << 20


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)


@pytest.fixture
def limit():
    """Sets the limit, from a state in which the library keeps nothing for later calls."""
    import paper_1102_1003_gb300 as pkg

    def set_to(nbytes):
        gc.collect()
        pkg.batmap_release_scratch()
        pkg.batmap_test_memory_limit(nbytes)

    yield set_to
    pkg.batmap_test_memory_limit(0)
    pkg.batmap_release_scratch()


def _inst(m, n, size, seed):
    rng = np.random.default_rng(seed)
    return datagen.from_lists([np.sort(rng.choice(m, size, replace=False)).astype(np.uint32) for _ in range(n)], m, s=1)


def _mine(inst, **params):
    """Supports against the merge oracle; returns the timing of the call."""
    import torch
    import paper_1102_1003_gb300 as pkg
    off, tids, _ = device_inputs(inst, 0)
    b = pkg.batmap_build(inst.m, off, tids, params=pkg.batmap_default_params(**params))
    full = torch.full((inst.n * (inst.n - 1) // 2,), -1, dtype=torch.int32, device="cuda")
    pkg.pair_support_all(b, 1, pairs=torch.empty((1, 3), dtype=torch.int32, device="cuda"), full=full)
    ref = oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS)
    assert np.array_equal(full.cpu().numpy().astype(np.uint32), ref)
    t = pkg.batmap_get_timing(b)
    b.free()
    return t


def test_idle_memory_is_given_back(limit):
    """BatMaps of 6.3 MB an item: the second set does not fit beside the first one's kept array,
    nor do a pool's arrays beside the second's."""
    import paper_1102_1003_gb300 as pkg
    params = dict(load_num=16, probe_log=32)
    a, b, c = _inst(1 << 20, 64, 1 << 17, 1), _inst(1 << 20, 75, 1 << 17, 2), _inst(1 << 20, 30, 1 << 17, 3)
    limit(700 * MB)
    _mine(a, **params)
    _mine(b, **params)
    off, tids, _ = device_inputs(c, 0)
    pool = pkg.batmap_pool_create(c.m, off, tids, params=pkg.batmap_default_params(load_num=16))
    qs = [[i, (i + 7) % c.n] for i in range(c.n)]
    assert np.array_equal(pkg.intersect_query(pool, qs).cpu().numpy().astype(np.uint64),
                          oracle.kway_counts(c.offsets, c.tids, qs))
    pool.free()


def test_no_memory_is_reported_once(limit):
    """A build that does not fit is refused as such, and the calls after it are not."""
    import paper_1102_1003_gb300 as pkg
    a = _inst(1 << 20, 64, 1 << 17, 1)
    off, tids, _ = device_inputs(a, 0)
    limit(50 * MB)
    with pytest.raises(pkg.BatmapError) as err:
        pkg.batmap_build(a.m, off, tids)
    assert err.value.code == pkg.BATMAP_ERR_NOMEM
    _mine(_inst(30_000, 40, 1_500, 4))
    pkg.batmap_test_memory_limit(0)
    _mine(a)


@pytest.mark.parametrize("d", [2, 3])
def test_equal_builds_take_equal_routes(limit, d):
    """Rows of 80 MB: less than half of what is free at first, more than half of what is left while
    the library keeps a freed set's arrays.  They are taken on every pass, or on none."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m, n = 1 << 22, 160
    inst = _inst(m, n, 200_000, 5)
    off, tids, _ = device_inputs(inst, 0)
    pairs = torch.tensor([[0, 1, 1], [0, 2, 1], [1, 2, 1]], dtype=torch.int32, device="cuda")
    want = int(oracle.kway_counts(inst.offsets, inst.tids, [[0, 1, 2]])[0])
    for room, rows in ((300 * MB, True), (150 * MB, False)):  # beside the BatMaps
        limit(n * (d + 1) * (1 << 19) + room)
        for _ in range(3):
            if d == 2:
                t = _mine(inst)
            else:
                b = pkg.batmap_build_d(d, m, off, tids)
                n_out, triples, n_cand = pkg.frequent_triples(b, 1, pairs)
                assert n_cand == 1 and triples.tolist() == [[0, 1, 2, want]]
                t = pkg.batmap_get_timing(b)
                b.free()
            assert (t["scan_ms"] == 0) == rows


@pytest.mark.parametrize("room,rows", [(180, False), (400, True)])
def test_rows_leave_room_for_the_supports(limit, room, rows):
    """67 MB of rows beside 122 MB of supports, for which the BatMap route has room in 180."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m, n = 70_001, 8_000
    inst = datagen.bernoulli_tidlists(m, n, 0.003, seed=7)
    off, tids, _ = device_inputs(inst, 0)
    limit(n * 3 * 1024 + room * MB)
    b = pkg.batmap_build(m, off, tids)
    n_out, pairs = pkg.pair_support_all(b, 3, pairs=torch.empty((n * n // 2, 3), dtype=torch.int32, device="cuda"))
    assert (pkg.batmap_get_timing(b)["scan_ms"] == 0) == rows
    b.free()
    ref = oracle.threshold_from_full(oracle.pairs_full(inst.offsets, inst.tids, threads=THREADS), n, 3)
    assert n_out == ref.shape[0] and np.array_equal(pairs.cpu().numpy().astype(np.uint32), ref)


def test_kept_arrays_are_bounded_in_bytes(limit):
    """Freed sets of several sizes: what the library keeps of them stays below a quarter of the
    memory (here of the limit), and an array above that is not kept."""
    import torch
    import paper_1102_1003_gb300 as pkg
    insts = [_inst(1 << 20, n, 1 << 17, n) for n in (14, 20, 30, 45, 68)]  # BatMaps of 84 to 408 MB
    for inst in insts:  # (the first calls of the process take memory of their own)
        _mine(inst, load_num=16, probe_log=32)
    limit(1_000 * MB)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = torch.cuda.mem_get_info()[0]
    for inst in insts:
        _mine(inst, load_num=16, probe_log=32)
    torch.cuda.empty_cache()
    kept = before - torch.cuda.mem_get_info()[0]
    # a quarter, the placement scratch (at most 96 MiB of regions here, and its tasks) and small arenas
    assert kept < (250 + 110 + 40) * MB
    assert kept > 80 * MB  # and the smaller ones are still kept
