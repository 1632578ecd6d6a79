"""The details of bench.py's line stay short: a batch's columns are summed up, not listed, and floats carry six digits."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


def test_columns_are_summed_up():
    import bench
    st = [{"iterations": 47 + i % 4, "true_relres": 9.123456789012345e-07 - 1e-10 * i, "converged": True, "est_relres": 1e-7}
          for i in range(128)]
    d = bench.short_floats(bench.columns_summary(st))
    assert d == {"iterations": [47, 50], "true_relres_max": 9.12346e-07, "converged": True}
    assert len(json.dumps(d)) < 100


def test_short_floats_leave_the_rest():
    import bench
    x = {"a": 1, "b": None, "c": True, "d": "1.23456789", "e": [1.0 / 3.0, 10, (2.0 / 3.0,)], "f": 31574708736.0}
    assert bench.short_floats(x) == {"a": 1, "b": None, "c": True, "d": "1.23456789", "e": [0.333333, 10, [0.666667]],
                                     "f": 31574700000.0}
