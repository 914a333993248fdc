"""Lists and permutation tables that a build refuses are refused soon: the check
runs beside the placement, whose chains of equal copies would otherwise take all
their moves (here 3 * 2^20 each, one exchange after the other: minutes)."""
import time

import numpy as np
import pytest

import datagen
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


@pytest.mark.parametrize("probe_log", [0, 32])  # lists checked by the bit rows' build, or by a kernel of its own
@pytest.mark.parametrize("d", [2, 3, 4])
@pytest.mark.parametrize("fault", ["small", "large", "table"])
def test_refused_without_the_chains(fault, d, probe_log):
    import torch
    import paper_1102_1003_gb300 as pkg
    m, rng = 1 << 18, np.random.default_rng(d)
    lists = [np.sort(rng.choice(m, s, replace=False)).astype(np.uint32) for s in [3_000] * 20 + [150_000] * 3]
    inst = datagen.from_lists(lists, m)
    off, tids, _ = device_inputs(inst, 0)
    perm = None
    if fault == "table":
        perm = torch.zeros((d + 1, m), dtype=torch.int32, device="cuda")
    else:  # every tid of an item the same: its table in shared memory, or in L2
        i = 7 if fault == "small" else 21
        tids[int(inst.offsets[i]):int(inst.offsets[i + 1])] = 5
    p = pkg.batmap_default_params(max_loop=1 << 20, probe_log=probe_log)
    torch.cuda.synchronize()
    t0 = time.monotonic()
    with pytest.raises(pkg.BatmapError) as err:
        pkg.batmap_build_d(d, m, off, tids, perm, params=p)
    assert err.value.code == pkg.BATMAP_ERR_ARG
    assert time.monotonic() - t0 < 5.0
