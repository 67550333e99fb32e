"""The benchmark's count of the kernels it starts."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_a_row_owner_pass_is_three_launches():
    """Geometry, bounds and assembly; FP64 takes the two forms one at a time."""
    assert bench.launches_of(("p3", [0, 1], "rows"), "fp32") == 3
    assert bench.launches_of(("p3", [0, 1], "rows"), "fp64") == 6
    assert [bench.launches_of(("p1", [0, 1], k), p) for k in ("pair", "single") for p in ("fp32", "fp64")] == [1, 2, 1, 1]
