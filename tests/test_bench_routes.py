"""bench.py without pair tables times the rank-code evaluator, which has to be asked for: a plain call
with a large population would build a pair table for itself."""
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_no_pairs_asks_for_the_evaluator():
    import bench
    from paper_1807_09932_gb300 import ebic
    assert bench.route_flags(True) == ebic.EBIC_EVAL_DIRECT
    assert bench.route_flags(False) == 0
