"""The benchmark names the sweep kernel that its workspace reports."""

import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_sweep_named_by_what_runs():
    import bench
    names = [bench.sweep_name({"sweep": s}, 64) for s in (0, 1, 2)]
    assert names == ["k_sweep<64>", "k_sweep_tma<64>", "k_tiles<64>"]
