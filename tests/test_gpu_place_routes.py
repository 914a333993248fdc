"""Placement in more than one chain of launches, and from a written-out table of
the computed permutations: every BatMap against the definition of the layout."""
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


# tables of 1.5 MB (the first also of 3 MB): chains of 62 to 64 of them fill the regions once, of 140 twice
@pytest.mark.parametrize("n", [62, 63, 64, 65, 140])
def test_chains_of_batches(n):
    import paper_1102_1003_gb300 as pkg
    m = 1 << 18
    inst = _items(m, [70_000] + [40_000 - 7 * i for i in range(n - 1)], seed=n)
    off, tids, _ = device_inputs(inst, 5)
    b = pkg.batmap_build(m, off, tids, params=seeded_params(5))
    assert layout_errors(inst, b, 5) == []


# 2^b / m from 1.6 to 3.99 and 1.5 - (computed); 16 m tids and just below; both homes of a table
@pytest.mark.parametrize("d", [2, 3, 4])
@pytest.mark.parametrize("m,size", [(40_000, 7_000), (4_105, 1_500), (10_923, 3_000), (10_922, 3_000), (70_000, 30_000)])
@pytest.mark.parametrize("less", [0, 1])
def test_table_of_computed_permutations(d, m, size, less):
    import paper_1102_1003_gb300 as pkg
    from oracle import dof_rules as R
    from oracle import permutation as OP
    sizes = [size] * (16 * m // size)
    sizes.append(16 * m - sum(sizes) - less)
    inst = _items(m, sizes, seed=m + less)
    off, tids, _ = device_inputs(inst, 5)
    if d == 2:
        b = pkg.batmap_build(m, off, tids, params=seeded_params(5))
        assert layout_errors(inst, b, 5) == []
        return
    b = pkg.batmap_build_d(d, m, off, tids, params=seeded_params(5))
    lay = pkg.batmap_export_layout(b)
    s, r0, perms = lay["info"]["shift"], lay["info"]["r0"], OP.permutations(m, 5, d + 1)
    for i in range(inst.n):
        r, at = int(lay["range"][i]), int(lay["byte_offset"][i])
        failed = lay["fail_tids"][int(lay["fail_offsets"][i]):int(lay["fail_offsets"][i + 1])]
        assert list(R.check_layout(lay["bytes"][at:at + (d + 1) * r], inst.tidlist(i), failed, perms, r, r0, s, d)) == []


# elements that cannot be placed: none, some, and more chains than the list of long ones holds
@pytest.mark.parametrize("load", [(2, 1), (1, 1), (1, 2)])
@pytest.mark.parametrize("max_loop", [5, 6, 32])  # 15, 18 and 96 moves, 16 before a chain waits
@pytest.mark.parametrize("m", [60_000, 4_096])
def test_long_chains_in_shared_memory(load, max_loop, m):
    import paper_1102_1003_gb300 as pkg
    inst = _items(m, [0, 1, 33, 1_000, 2_047, 4_000, 4_096, 4_096], seed=max_loop)
    off, tids, _ = device_inputs(inst, 5)
    b = pkg.batmap_build(m, off, tids, params=seeded_params(5, pkg.batmap_default_params(
        load_num=load[0], load_den=load[1], max_loop=max_loop)))
    assert layout_errors(inst, b, 5, *load) == []
