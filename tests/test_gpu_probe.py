"""The three ways in which a task's elements are looked up in another set (read
side by side, searched, byte probes), at the ends of rows (32), parts and tasks
(512) and of the ratio of sizes that separates them, at every alignment of the
lists, for disjoint, nested and equal sets: lists and counts against numpy."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,universe", [(1 << 16, 1 << 16), (1 << 24, 300_000), (1 << 30, 300_000)])
@pytest.mark.parametrize("shift", [0, 1, 2, 3])
def test_lists_by_size_and_alignment(m, universe, shift):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    import paper_1102_1003_gb300 as pkg
    torch.cuda.set_device(0)
    rng = np.random.default_rng(universe + shift)
    u = np.unique(np.concatenate([[0, m - 1], rng.choice(m, universe, replace=False)])) if universe < m else np.arange(m)
    sizes = [s for s in (shift, 0, 1, 2, 31, 32, 33, 511, 512, 513, 1025, 2000, 16_383, 16_385, 40_000, 140_000) if s <= u.size]
    sets = [np.sort(rng.choice(u, s, replace=False)) for s in sizes]
    # neighbouring runs: below, above, inside and the same
    sets += [u[100:700], u[700:1300], u[50:2000:3], u[-600:], u[:600], u[100:700]]
    off = np.concatenate([[0], np.cumsum([s.size for s in sets])]).astype(np.int64)
    tids = np.concatenate(sets).astype(np.int32)
    pool = pkg.batmap_pool_create(m, torch.from_numpy(off).cuda(), torch.from_numpy(tids).cuda())
    n = len(sets)
    queries = [[i, j] for i in range(n) for j in range(i, n)] + [[i] for i in range(n)]
    queries += [rng.integers(0, n, k).tolist() for k in range(3, 9) for _ in range(20)]

    def common(q):
        out = sets[q[0]]
        for i in q[1:]:
            out = np.intersect1d(out, sets[i])
        return out

    want = [common(q) for q in queries]
    ends, got = pkg.intersect_query_list(pool, queries)
    assert np.array_equal(ends.cpu().numpy(), np.concatenate([[0], np.cumsum([w.size for w in want])]))
    assert np.array_equal(got.cpu().numpy(), np.concatenate(want))
    assert np.array_equal(pkg.intersect_query(pool, queries).cpu().numpy(), [w.size for w in want])
