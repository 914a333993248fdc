"""Placement of 3-of-4 and 4-of-5 sets whose tables fill the larger regions of L2: two
sequences of batches of 16 items, with and without a caller's permutation table.  Every
BatMap against the definition of the layout."""
import numpy as np
import pytest

import datagen
from oracle import dof_rules as R
from oracle import permutation as OP

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    torch.cuda.set_device(0)


# tables of 2.1 (d = 3) and 2.6 MB: from 64 of them on a region holds 16, below it holds fewer
@pytest.mark.parametrize("d", [3, 4])
@pytest.mark.parametrize("n", [63, 64, 65, 100])
@pytest.mark.parametrize("table", [False, True])
def test_regions_of_sixteen_items(d, n, table):
    import torch
    import paper_1102_1003_gb300 as pkg
    m = 1 << 18
    rng = np.random.default_rng(n)
    inst = datagen.from_lists([np.sort(rng.choice(m, 65_000 - 7 * i, replace=False)).astype(np.uint32) for i in range(n)], m)
    off = torch.from_numpy(inst.offsets.astype(np.int64)).cuda()
    tids = torch.from_numpy(inst.tids.astype(np.int32)).cuda()
    perms = datagen.permutations(m, 3, count=d + 1) if table else OP.permutations(m, 3, d + 1)
    p = torch.from_numpy(perms.astype(np.int32)).cuda() if table else None
    b = pkg.batmap_build_d(d, m, off, tids, p, params=pkg.batmap_default_params(perm_seed=3))
    lay = pkg.batmap_export_layout(b)
    s, r0 = lay["info"]["shift"], lay["info"]["r0"]
    for i in range(inst.n):
        r, at = int(lay["range"][i]), int(lay["byte_offset"][i])
        assert r == 1 << 17
        failed = lay["fail_tids"][int(lay["fail_offsets"][i]):int(lay["fail_offsets"][i + 1])]
        assert list(R.check_layout(lay["bytes"][at:at + (d + 1) * r], inst.tidlist(i), failed, perms, r, r0, s, d)) == []
