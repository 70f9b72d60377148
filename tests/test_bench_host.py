"""Host-side pieces of bench.py that need no GPU: the traffic table keyed on the head kernel's
sources."""
import bench


def test_traffic_table_is_from_one_capture_of_the_sources():
    hashes = {h for (_, h) in bench.HEAD_TRAFFIC}
    assert len(hashes) == 1
    assert all(v > 1e9 for v in bench.HEAD_TRAFFIC.values())
    assert len(bench.head_source_hash()) == 16
