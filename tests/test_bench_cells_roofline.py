"""The benchmark's roofline of the matching through cells: figures counted on one captured workload are given for that
workload only."""
import pytest

import bench


@pytest.mark.parametrize("sizes,captured", [((3, 256, 2048, 8192), True), ((1, 32, 256, 512), False), ((3, 1024, 4096, 65536), False)])
def test_captured_figures_stay_with_their_workload(sizes, captured):
    entry = bench.cells_roofline_entry(sizes, 40e-6, [40.0, 20.0, 15.0, 25.0, 10.0, 0.0], 152, {"sm_mhz": 2000.0})
    P, K, N, M = sizes
    assert entry["queries_per_launch"] == P * K * N and entry["pairs_per_launch"] == P * K * N * M
    assert entry["achieved"] == pytest.approx(P * K * N / 40e-6 / 1e9)
    assert (entry["traffic"] is not None) == captured
    assert (entry["frac"] is not None) == captured and (entry["peak"] is not None) == captured
    if captured:
        assert entry["peak"] == pytest.approx(152 * 128 * 2e9 / bench.CELLS_LANE_INST_PER_QUERY / 1e9)
        assert entry["frac"] == pytest.approx(entry["achieved"] / entry["peak"])
