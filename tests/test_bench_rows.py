"""Roofline rows of bench.py: a launch that is a whole CG loop has no product bandwidth."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_product_launches_have_a_bandwidth():
    import bench
    r = bench.kernel_row("spmv", 2_000_000, 1.0, 100, 500.0, products=90)   # 100: with idle launches
    assert r["kernel"] == "spmv" and r["bytes_per_launch"] == 2_000_000
    assert r["us_per_launch"] == pytest.approx(10.0)
    assert r["achieved_gbs"] == pytest.approx(200.0) and r["frac"] == pytest.approx(0.4)


def test_whole_loops_have_none():
    import bench
    r = bench.kernel_row("spmv", 2_000_000, 10.0, 4, 500.0, products=400)
    assert "k_cg_loop" in r["kernel"] and "100.0" in r["kernel"]
    assert r["us_per_launch"] == pytest.approx(2500.0) and r["launches"] == 4
    assert r["achieved_gbs"] is None and r["frac"] is None and r["bytes_per_launch"] is None


def test_no_launch():
    import bench
    r = bench.kernel_row("spmv", 1, 0.0, 0, 500.0, products=0)
    assert r["us_per_launch"] is None and r["frac"] is None
