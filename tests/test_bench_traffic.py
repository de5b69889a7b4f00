"""The bench reports captured DRAM traffic only for the sources it was captured on (no GPU needed)."""
import bench


def test_recorded_traffic_belongs_to_the_current_sources():
    stale = [name for name in bench.NCU_TRAFFIC if bench.ncu_traffic(name) is None]
    assert not stale, f"captured on other sources: {stale}"
    assert set(bench.NCU_TRAFFIC) <= set(bench.KERNEL_SOURCES)
