"""bench.py measures the FP64 near field against what bounds it."""
import os
import sys

import pytest

pytest.importorskip("torch")
sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def test_fp64_near_field_rate_is_a_fraction_of_a_limit():
    """421 million body pairs in 7.2 ms (a Plummer sphere of 1,048,576): each from both
    sides, 36 products a side, of 31.6 per clock and SM."""
    achieved, limit = bench.p2p64_rate(421_000_000, 7.2)
    assert achieved == pytest.approx(2 * 421e6 * 36 / 7.2e-3 / 1e12)
    assert limit == pytest.approx(152 * 2070e6 * 31.6 / 1e12)
    assert 0.3 < achieved / limit < 1.0
