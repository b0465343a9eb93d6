"""bench.py's FP64 roofline: the fraction is of what the pipe executes.

The formulation's flops, about half of which run as integers, are reported as a rate
beside it, which may exceed the pipe's peak.
"""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402


def test_pipe_fraction_counts_executed_instructions():
    pts, ms, peak = 128 ** 3, 0.2578, 1.2556
    r = bench.roofline_for("fp64", pts, ms, 6789.3, fp64_measured=peak)
    p = r["fp64_pipe"]
    assert p["instructions_per_point"] < bench.FP64_FLOP_PER_POINT / 2
    assert p["achieved"] == pytest.approx(58 * pts / (ms * 1e-3) / 1e12)
    assert p["peak"] == pytest.approx(peak / 2) and p["frac"] == pytest.approx(p["achieved"] / p["peak"])
    assert p["frac"] < 1.0 < r["frac"]
    line = {"value": 1.0, "ms_per_step": ms, "roofline": r, "variants": {}}
    assert bench.summary(line)["headline"]["frac"] == p["frac"]
