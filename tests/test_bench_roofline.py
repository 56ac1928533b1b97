"""bench.py's roofline of the recursion: a fraction of the rate that the products of the
kernel that ran it have."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402


@pytest.mark.parametrize("prec,column,peak,kernel", [
    ("f32", True, 604.0 / 6, "k_colstep<float>"), ("f64", True, 604.0 / 26, "k_colstep<double>"),
    ("f64x", True, 604.0 / 26, "k_colstep<double>"), ("f32", False, 80.56, "k_resident<float>"),
    ("f64", False, 1.26, "k_step<double>"), ("f64x", False, 80.56, "k_step<dfl>"),
])
def test_the_peak_is_that_of_the_kernel(prec, column, peak, kernel):
    tflops = 0.6 if prec == "f64" and not column else 5.3  # (measured ones: four times the FP64 unit by digits)
    roof = bench.step_roof(tflops, prec, column)
    assert roof["peak"] == pytest.approx(peak, rel=1e-3) and roof["kernel"] == kernel
    assert roof["frac"] == pytest.approx(tflops / peak, rel=2e-3) and roof["frac"] < 1.0
    assert roof["bound"] == ("tensor" if column else "alu")
    key, unit = ("vs_fp32_unit_peak", 80.56) if prec == "f32" else ("vs_fp64_unit_peak", 1.26)
    assert roof[key] == pytest.approx(tflops / unit, rel=1e-3)
