"""Prefix sums over the tasks of a call at the border between one block (8,192
values) and tiles with look-back (2,048 values each): lists of as many queries
of one task each, against numpy; exact, as counts are integers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nq", [1, 2047, 8191, 8192, 8193, 10240, 10241, 70001])
def test_offsets_of_many_tasks(nq):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_1102_1003_gb300 as pkg
    torch.cuda.set_device(0)
    m, n = 1000, 40
    rng = np.random.default_rng(nq)
    sets = [np.sort(rng.choice(m, 1 + 5 * i, replace=False)).astype(np.int32) for i in range(n)]
    off = np.concatenate([[0], np.cumsum([s.size for s in sets])]).astype(np.int64)
    pool = pkg.batmap_pool_create(m, torch.from_numpy(off).cuda(), torch.from_numpy(np.concatenate(sets)).cuda())
    pairs = rng.integers(0, n, (nq, 2))
    common = {(a, b): np.intersect1d(sets[a], sets[b]) for a in range(n) for b in range(n)}
    want = [common[a, b] for a, b in pairs.tolist()]
    got_off, got = pkg.intersect_query_list(pool, pairs.tolist())
    assert np.array_equal(got_off.cpu().numpy(), np.concatenate([[0], np.cumsum([w.size for w in want])]))
    assert np.array_equal(got.cpu().numpy(), np.concatenate(want))
