"""The committed profile of the FP32 step is of the kernel in the tree: bench.py
reports its DRAM traffic only while the hash of the sources matches."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402


def test_the_profile_is_of_this_kernel():
    b = bench.profiled_traffic(7)
    assert b is not None
    # 216 B of populations a cell, at most 2 % more
    assert 0.98 <= b / (216 * 4096 * 4096) <= 1.02
