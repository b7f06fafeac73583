"""Arithmetic of the bench's roofline entries (no GPU needed)."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))


@pytest.mark.parametrize("launches", [1, 22])
def test_rate_is_of_the_whole_phase(launches):
    """6e12 operations in 3 ms of a build are 2000 TFLOP/s, in however many launches."""
    import bench
    r = bench.roofline_of({"k": (3.0, launches)}, "k", flops=6e12, peak=2500.0)
    assert r["achieved"] == pytest.approx(2000.0) and r["frac"] == pytest.approx(0.8)
    r = bench.roofline_of({"k": (3.0, launches)}, "k", nbytes=6e9, peak=8000.0, bound="hbm", unit="GB/s")
    assert r["achieved"] == pytest.approx(2000.0)
    assert bench.roofline_of({}, "k", flops=1.0, peak=1.0) is None


@pytest.mark.parametrize("m,n,k", [(129, 33, 33), (1500, 1500, 4500 * 15), (40, 16, 32), (600, 60, 600)])
def test_issued_operations_cover_the_contraction(m, n, k):
    import bench
    dense = bench.DIGIT_PRODUCTS * 2.0 * m * n * k
    pad = (-(-m // 128) * 128 / m) * (-(-n // 64) * 64 / n) * (-(-k // 32) * 32 / k)
    assert dense <= bench.digit_gemm_flops(m, n, k) <= dense * pad * (1 + 1e-12)
    if m == n:  # the lower triangle in tiles: more than half, less than all
        assert dense / 2 <= bench.digit_gemm_flops(m, n, k, lower=True) < bench.digit_gemm_flops(m, n, k)
