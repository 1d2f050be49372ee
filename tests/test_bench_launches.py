"""The launch count of the bench line: it follows the form that the handle says
it runs, not a size of its own."""
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_launches_follow_the_handles_form():
    sys.path.insert(0, ROOT)
    import bench
    assert bench.launches_per_solve(500, False) == 9 + 3 * 500
    assert bench.launches_per_solve(500, True) == 10
