"""Pools take hash ranges below the 2^7 that batmap_build asks for: BatMaps of 3
bytes and more, whose neighbours start at any byte.  Counts against the merge
oracle, exact."""
import numpy as np
import pytest

import datagen
import oracle
from tests.gpu_util import device_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)


# load 1/50: more elements than slots, so that their tables go to L2; 16/1: wide tables beside narrow ones
@pytest.mark.parametrize("load", [(2, 1), (16, 1), (1, 50)])
@pytest.mark.parametrize("min_shift", [0, 1, 3, 6])
@pytest.mark.parametrize("m", [1, 100, 127, 1_000, 9_000])
def test_narrow_batmaps(m, min_shift, load):
    import paper_1102_1003_gb300 as pkg
    rng = np.random.default_rng(m + min_shift)
    sizes = np.concatenate([np.full(12, 1), np.minimum(m, rng.integers(1, 40, 12)), rng.integers(1, m + 1, 12), [m, m]])
    inst = datagen.from_lists([np.sort(rng.choice(m, s, replace=False)).astype(np.uint32) for s in sizes], m)
    off, tids, _ = device_inputs(inst, 0)
    p = pkg.batmap_default_params(min_shift=min_shift, load_num=load[0], load_den=load[1], max_loop=3)
    pool = pkg.batmap_pool_create(m, off, tids, params=p)
    qs = [[int(a), int(b)] for a in range(inst.n) for b in range(inst.n)] + rng.integers(0, inst.n, (200, 4)).tolist()
    got = pkg.intersect_query(pool, qs).cpu().numpy().astype(np.uint64)
    assert np.array_equal(got, oracle.kway_counts(inst.offsets, inst.tids, qs))
    if load == (2, 1) and min_shift == 0 and m == 100:
        assert pool.info["n_batmaps"] == inst.n  # even the sets of one element (r = 2: 6 bytes)


def test_chains_end_whatever_max_loop():
    """max_loop of a pool is not limited; an element that cannot be placed (20 copies, 12 slots) is
    given up all the same and found by its list."""
    import paper_1102_1003_gb300 as pkg
    lists = [np.arange(0, 100, 10), np.arange(0, 120, 12), np.arange(60), np.arange(0, 127, 2)]
    inst = datagen.from_lists([x.astype(np.uint32) for x in lists], 127)
    off, tids, _ = device_inputs(inst, 0)
    p = pkg.batmap_default_params(min_shift=0, load_num=1, load_den=3, max_loop=1 << 30)
    pool = pkg.batmap_pool_create(127, off, tids, params=p)
    qs = [[a, b] for a in range(4) for b in range(4)]
    got = pkg.intersect_query(pool, qs).cpu().numpy().astype(np.uint64)
    assert np.array_equal(got, oracle.kway_counts(inst.offsets, inst.tids, qs))


@pytest.mark.parametrize("tasks", [1, 255, 256, 257, 600])
def test_tasks_from_the_host_and_from_the_device(tasks):
    """Batches of up to 256 tasks bring them along, larger ones make them on the device; counts,
    lists and the serving loop agree with merges on either side."""
    import paper_1102_1003_gb300 as pkg
    m, rng = 40_000, np.random.default_rng(tasks)
    sizes = [0, 1, 127, 128, 129, 511, 512, 513, 3_000, 9_000, 20_000]  # around a task's and a chunk's end
    inst = datagen.from_lists([np.sort(rng.choice(m, s, replace=False)).astype(np.uint32) for s in sizes], m)
    off, tids, _ = device_inputs(inst, 0)
    pool = pkg.batmap_pool_create(m, off, tids)
    # tasks of 128 elements (small batches): as many queries on the sets of up to 128 as there are tasks
    qs = [[int(rng.integers(1, 4)), int(rng.integers(1, len(sizes)))] for _ in range(tasks)]
    for batch in (qs, qs + [[0, 9], [9, 10], [10, 8, 9], [4, 5], [6], [7, 6, 10]]):
        want = oracle.kway_counts(inst.offsets, inst.tids, batch)
        assert np.array_equal(pkg.intersect_query(pool, batch).cpu().numpy().astype(np.uint64), want)
        o, elems = pkg.intersect_query_list(pool, batch)
        o, elems = o.cpu().numpy(), elems.cpu().numpy().astype(np.uint32)
        assert np.array_equal(np.diff(o).astype(np.uint64), want)
        for q, ids in enumerate(batch):
            both = inst.tidlist(ids[0])
            for i in ids[1:]:
                both = np.intersect1d(both, inst.tidlist(i), assume_unique=True)
            assert np.array_equal(elems[o[q]:o[q + 1]], both)
        opts = pkg.batmap_serve_opts(max_batch=tasks, slots=3, work_budget=1 << 26, reserved=0)
        counts, _, _ = pkg.batmap_serve(pool, batch, np.zeros(len(batch)), opts)
        assert np.array_equal(np.asarray(counts, np.uint64), want)
