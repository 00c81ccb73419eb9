"""bench.py's count of kernel launches and the kernel it names follow what the
solver reports: every driver that AUTO can choose."""
import pytest

import bench

CASES = [  # mode, cluster, launches per iteration: launches of 200 iterations, kernel
    ("resident", 1, 0, 1, "hs_resident_kernel"),
    ("persistent", 4, 0, 2, "hs_persistent_kernel"),
    ("persistent", 0, 0, 2, "hs_narrow_kernel"),
    ("queue", 1, 0, 2, "hs_queue_kernel"),
    ("warp", 1, 0, 2, "hs_warp_kernel"),
    ("looped", 2, 19, 3800, "hs_looped_kernel"),
    ("structured", 1, 4, 800, "struct_kernel"),
    ("structured", 1, 0, 2, "struct_queue_kernel"),
    ("structured_queue", 1, 0, 2, "struct_queue_kernel"),
]


@pytest.mark.parametrize("mode,cluster,per_iteration,launches,kernel", CASES)
def test_launches_and_kernel(mode, cluster, per_iteration, launches, kernel):
    info = {"mode": mode, "cluster": cluster, "launches_per_iteration": per_iteration, "phases": 19}
    assert bench.run_launches(info, 200) == launches
    assert bench.run_kernel(info) == kernel
