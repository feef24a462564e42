"""The bench line's roofline entry of the fixed-point FP64 operator (host arithmetic, CPU): the fraction is of the integer
multiply-add rate, the FP64 unit's figures stand apart."""
import pytest

import bench


def test_fixed_point_operator_entry_by_hand():
    e = bench.roofline_entry("fp64_operator", 64, 7, 0.0966, 32 ** 3, 859812, 152, 2070.0, 1.056,
                             {"bf16_tflops": 1912.0, "hbm_gbs": 6777.6}, "not-the-sources", 5)
    # a thread's products: 60 + 60 + 180 (interpolation), 297 (A), 108 (B^T), 90 (B), 36 (pressure), 189 + 108 (transposes),
    # 36 (pressure sums)
    mads = 9 * (60 + 60 + 180 + 297 + 108 + 90 + 36 + 189 + 108 + 36) * 32 ** 3
    assert e["int_mads_per_launch"] == mads
    assert e["achieved"] == pytest.approx(mads / 0.0966e-3 / 1e12, abs=1e-4)
    assert e["peak"] == pytest.approx(152 * 50 * 2.07e9 / 1e12, abs=1e-4)
    assert e["frac"] == pytest.approx(mads / 0.0966e-3 / (152 * 50 * 2.07e9), abs=1e-4) and e["frac"] < 1
    fp64 = e["fp64_unit_comparison"]
    assert fp64["frac"] == pytest.approx(12768 * 32 ** 3 / 0.0966e-3 / 1e12 / 1.25856, abs=1e-4)
    assert "frac_of_peak_from_measured_bf16" not in e and e["traffic"] is None
