"""The bench's captured DRAM figures: reported only for what they were taken on (no GPU)."""
import os
import re


def test_captured_traffic_needs_the_launch_shape_it_was_taken_with():
    """DRAM bytes of a capture are reported for its sources, workload and launch shape only."""
    import bench
    tr = {"bytes": 7, "hash": "h", "workload": "w", "taken_with": bench.DEFAULT_SHAPE}
    assert bench.captured_traffic(tr, "h", "w") == 7                      # untuned run
    assert bench.captured_traffic(tr, "h", "w", dict(bench.DEFAULT_SHAPE, source="--tune")) == 7
    assert bench.captured_traffic(tr, "h", "w", {"lpc": 1, "chunk_bytes": 64 << 20, "row_variant": 0}) is None
    assert bench.captured_traffic(tr, "h", "w", {"lpc": 2, "chunk_bytes": 512 << 20, "row_variant": 0}) is None
    assert bench.captured_traffic(tr, "g", "w") is None and bench.captured_traffic(tr, "h", "v") is None
    assert bench.captured_traffic(None, "h", "w") is None
    assert bench.captured_traffic({"bytes": 3, "hash": "h", "workload": "w"}, "h", "w", {"lpc": 2}) == 3
    # every file a stage is built from is part of its hash
    for files in (bench.GATHER_SOURCES, bench.GRID_SOURCES, bench.DIRECT_SOURCES):
        for name in files:
            text = open(os.path.join(bench.ROOT, "paper_2005_12716_gb300", name), encoding="utf-8").read()
            for inc in re.findall(r'#include "(\w+\.cuh)"', text):
                assert "csrc/" + inc in files, (files[0], inc)
