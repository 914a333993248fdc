"""What the bench says about a step fits the route that it took (CPU only): no bandwidth
of BatMaps that the contraction of bit rows does not read, no schedule tuned for nothing."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402

PEAKS = {"hbm_gbs": 6761.6, "bf16_tflops": 1896.9}


def test_bandwidth_is_of_the_route_that_ran():
    m, n = 4_194_304, 8_192
    npairs = n * (n - 1) // 2
    word_pairs = npairs * 3 * 2**19 / 4
    rows = bench.route_keys(True, m, n, npairs, word_pairs, 0.0544, PEAKS)
    assert rows["dtype"] == bench.CONTRACT_DTYPE and "logical_hbm" not in rows
    assert 0 < rows["hbm"]["frac"] < 1  # 4.4 GB in 54.4 ms
    scan = bench.route_keys(False, m, n, npairs, word_pairs, 1.87, PEAKS)
    assert scan["dtype"] == "u8" and "hbm" not in scan
    assert abs(scan["logical_hbm"]["achieved_GBps"] - 8.0 * word_pairs / 1.87 / 1e9) < 1.0


def test_batmap_leg_only_beside_the_bit_rows():
    assert bench.batmap_leg(None, None, PEAKS, "", "", {"dtype": "u8"}) is None
