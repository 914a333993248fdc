"""The single-pass threshold compaction at the ends of its tiles (4,096
supports) and stages (2,048 triples), on supports of the test's own, against
numpy: exact, as supports are integers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)


def _want(full, n, s):
    i, j = np.triu_indices(n, 1)
    keep = full >= s
    return np.stack([i[keep], j[keep], full[keep]], 1)


# n(n-1)/2: 1, 4095, 4186, 8128, 8256, 40_470, 1_124_250
@pytest.mark.parametrize("n", [2, 3, 91, 92, 128, 129, 285, 1500])
@pytest.mark.parametrize("kind", ["none", "all", "some", "ends"])
@pytest.mark.parametrize("shift", [0, 1])
def test_triples_of_given_supports(n, kind, shift):
    import torch
    import paper_1102_1003_gb300 as pkg
    npairs = n * (n - 1) // 2
    rng = np.random.default_rng(n)
    full = rng.integers(0, 100, npairs)
    s = {"none": 1000, "all": 0, "some": 60, "ends": 1000}[kind]
    if kind == "ends":
        full[[0, npairs - 1]] = 2000
        full[np.arange(4095, npairs, 4096)] = 3000
    buf = torch.zeros(npairs + shift, dtype=torch.int32, device="cuda")
    buf[shift:] = torch.from_numpy(full.astype(np.int32)).cuda()  # shift 1: not on a 16-byte boundary
    want = _want(full, n, s)
    for cap in sorted({0, 1, max(0, len(want) - 1), len(want), len(want) + 3}):
        out = torch.full((cap + 2, 3), -1, dtype=torch.int32, device="cuda")
        k = pkg.pair_threshold_noalloc(buf[shift:], n, s, out[:cap] if cap else None)
        assert k == len(want)
        got = out.cpu().numpy()
        m = min(cap, len(want))
        assert np.array_equal(got[:m], want[:m]) and (got[m:] == -1).all()
