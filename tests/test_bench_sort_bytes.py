"""The benchmark's lines count for the sort what it moves (no GPU)."""
import ast
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_sort_bytes_of_the_two_launch_sort():
    # keys and places: x, y, z (24) in, key and index (12) out; the buckets' sort: key and index in and out (24)
    out = bench.hbm_stages(1 << 24, 8, {"sort": 6.6}, sort_bytes=bench.SORT_BYTES)["sort"]
    assert out["bytes_per_particle"] == 24 + 12 + 24
    assert out["GB/s"] == pytest.approx((1 << 24) * 60 * 8 / 6.6e-3 / 1e9)


def test_every_line_is_made_with_them():
    tree = ast.parse(open(os.path.join(ROOT, "bench.py")).read())
    calls = [c for c in ast.walk(tree) if isinstance(c, ast.Call) and getattr(c.func, "id", "") == "hbm_stages"]
    assert len(calls) == 2
    for c in calls:
        assert len(c.args) == 5 and c.args[4].id == "SORT_BYTES"
