"""Placement at the borders of its two homes (one CTA's shared memory up to
8,192 slots a table, L2 above): every BatMap is checked against the definition
of the layout (a tid in exactly two of its three slots, code and indicator,
empty slots 0, failed insertions listed), so nothing is compared inexactly."""
import numpy as np
import pytest

import datagen
from tests.gpu_util import device_inputs, layout_errors, seeded_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)


def _items(m, sizes, seed):
    rng = np.random.default_rng(seed)
    return datagen.from_lists([np.sort(rng.choice(m, s, replace=False)).astype(np.uint32) for s in sizes], m)


# sizes about the ends of warps, rounds, tasks (1,024 elements) and ranges (r doubles past a power of
# two); 4,096 fill the widest table in shared memory, 4,097 the first in L2
SIZES = [0, 1, 31, 32, 33, 127, 128, 129, 1023, 1024, 1025, 2048, 2049, 4095, 4096, 4097, 8191, 8192, 8193, 20_000]


@pytest.mark.parametrize("table", [False, True])
@pytest.mark.parametrize("params,m", [({}, 60_000), ({}, 200_001), (dict(load_num=1, load_den=4, max_loop=2), 60_000),
                                      (dict(load_num=16, load_den=1), 60_000)])
def test_layout_by_size(params, m, table):
    import paper_1102_1003_gb300 as pkg
    inst = _items(m, SIZES, seed=m + len(params))
    off, tids, perm = device_inputs(inst, 3, table)
    b = pkg.batmap_build(m, off, tids, perm, params=seeded_params(3, pkg.batmap_default_params(**params)))
    load = (params.get("load_num", 2), params.get("load_den", 1))
    assert layout_errors(inst, b, 3, *load, table=table) == []


def test_more_batches_than_epochs():
    """m = 2^30 leaves two bits for the epoch above a tid: the regions are cleared between
    batches.  Supports by the BatMap scan, which reads every byte."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m, n = 1 << 30, 9
    rng = np.random.default_rng(4)
    common = rng.choice(m, 300, replace=False)
    inst = datagen.from_lists([np.unique(np.concatenate([common, rng.choice(m, 500 * (i + 1))])).astype(np.uint32)
                               for i in range(n)], m)
    off, tids, _ = device_inputs(inst, 0)
    b = pkg.batmap_build(m, off, tids, params=pkg.batmap_default_params(probe_log=32))
    full = torch.zeros(n * (n - 1) // 2, dtype=torch.int32, device="cuda")
    pkg.pair_support_all(b, 1, full=full)
    want = [np.intersect1d(inst.tidlist(i), inst.tidlist(j)).size for i in range(n) for j in range(i + 1, n)]
    assert full.tolist() == want
    b.free()
    pkg.batmap_release_scratch()


def test_tids_out_of_range_are_skipped_without_validation():
    """validate = 0: tids >= m are left out, in both homes of the table."""
    import torch
    import paper_1102_1003_gb300 as pkg
    m = 60_000
    inst = _items(m, [500, 9_000], seed=1)
    lists = [np.concatenate([inst.tidlist(i), np.array([m, m + 5, 1 << 30], np.uint32)]) for i in range(2)]
    bad = datagen.from_lists(lists, m)
    off, tids, _ = device_inputs(bad, 0)
    b = pkg.batmap_build(m, off, tids, params=pkg.batmap_default_params(validate=0, probe_log=32))
    full = torch.zeros(1, dtype=torch.int32, device="cuda")
    pkg.pair_support_all(b, 1, full=full)
    assert full.tolist() == [np.intersect1d(inst.tidlist(0), inst.tidlist(1)).size]
