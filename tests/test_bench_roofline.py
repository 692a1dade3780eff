"""bench.py reports a roofline time for solves only where the work per pair is known."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench


def test_no_roofline_time_with_fp64_evaluations():
    rates = {"dfma_per_s": 6e11} if "dfma_per_s" in bench.eval_roofline_seconds.__code__.co_varnames else {}
    assert bench.eval_roofline_seconds((1e9, 0, 0), 152, 2070.0, **rates) is None
    assert bench.eval_roofline_seconds((1e9, 1e9, 1e9), 152, 2070.0, **rates) is None


def test_mixed_and_compensated_pairs():
    clk = 152 * 2070e6
    t = bench.eval_roofline_seconds((0, 1e9, 2e9), 152, 2070.0)
    assert t == pytest.approx(2e9 / (32 * clk) + 2e9 * 103 / (128 * clk))
