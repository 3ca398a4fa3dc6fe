"""The counts of executed flops (opcount.py)."""
import pytest

from paper_1408_7069_gb300 import opcount


def test_the_eigensolve_count_takes_sweeps():
    """Two slopes per cell, both triangles; 3.5 mp^3 per sweep; 10 mp^2 for the transform."""
    want = 868 * (4 * 32 ** 2 * 16 + 5.75 * 3.5 * 32 ** 3 + 10 * 32 ** 2)
    assert opcount.frame_executed_flops(32, 868, 16, 5.75) == pytest.approx(want)
    assert opcount.frame_executed_flops(32, 868, 16, mean_sweeps=5.75) == pytest.approx(want)


def test_the_series_count_takes_products():
    want = 868 * (4 * 32 ** 2 * 16 + 14 * 4 * 32 ** 2)
    assert opcount.frame_series_flops(32, 868, 16, mean_products=14) == pytest.approx(want)
    assert opcount.chebyshev_products(3.0) < opcount.chebyshev_products(30.0) < 100
