"""The benchmark's byte model of the rebalancing selection."""
import bench


def test_selection_bytes():
    work = {"select_levels": 5, "rebalance_evaluated": 1000}
    assert bench.selection_bytes(work, 4097 * 8, 8) == 16 * 4 * 1000  # read per level after the first
    assert bench.selection_bytes(work, 4096 * 8, 8) == 16 * 1000     # held in registers
