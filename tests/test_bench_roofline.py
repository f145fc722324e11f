"""The roofline's parts: FP64 flops and fixed-point operations of the committed
summary are kept apart, and the fixed-point rate of the GPU is that of its
products and sums in their mix."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_fixed_point_peak_is_the_rate_of_the_mix():
    assert bench.fixed_point_peak(10, 0, 152, 2000.0) == pytest.approx(7.5 * 152 * 2e9)
    assert bench.fixed_point_peak(0, 10, 152, 2000.0) == pytest.approx(42.0 * 152 * 2e9)
    # 75 products and 42 sums take 11 cycles of an SM
    assert bench.fixed_point_peak(75, 42, 1, 1.0) == pytest.approx(117 / 11 * 1e6)


def test_the_summary_keeps_fp64_and_fixed_point_apart():
    prof = bench.profiled(6_795_002, "k_flux + k_flux_hard<Euler,M=2>")
    assert prof["executed_flops_per_cell_update"] == pytest.approx(prof["fp64_flops"] + 2 * prof["products"] + prof["sums"])
    assert 0 < prof["fp64_flops"] < 30 and 80 < prof["products"] < 90
