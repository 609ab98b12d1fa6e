"""Launch counts that bench.py reports, against the launches that one evaluation
makes (counted from the launch code: preparation, recursions, exterior forces)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench


@pytest.mark.parametrize("N,precision,recompute,launches", [
    (16, "mixed", False, 3), (128, "fp64", True, 3), (128, "mixed32", False, 4), (129, "fp64", False, 4),
    (1024, "mixed", False, 4), (1792, "mixed", False, 4),       # 28 panels: one launch of the clusters
    (1793, "mixed", False, 6),                                  # two, one update between them
    (1025, "fp64", True, 6),
    (4096, "fp64", False, 12),                                  # four, three updates between, two beside
    (16384, "mixed", False, 48),                                # sixteen: 15 between, 14 beside
])
def test_launches_of_one_evaluation(N, precision, recompute, launches):
    assert bench.launches_per_eval(N, precision, recompute) == launches
