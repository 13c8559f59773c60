"""bench.py names the frame kernel and counts the launches from what the plan
runs on, not from the schedule's walk value (under which a small batch runs on
the segmented kernel alone)."""
import pytest

import bench


@pytest.mark.parametrize("walked,joints,kernel,launches", [
    (0, 1000, "k_scan_qt<0>", 2), (1000, 1000, "k_walk2", 2), (999, 1000, "k_walk2", 3), (100, 1000, "k_scan_qt<0>", 3)])
def test_frame_kernels(walked, joints, kernel, launches):
    name, n = bench.frame_kernels(walked, joints)
    assert name.startswith(kernel) and n == launches
