"""The roof that bench.py sets a kernel against: the fixed-point transforms of the
FP64 form never against the FP64 pipe, however near its rate their flops come; its
pointwise kernels and the one-line z passes in doubles against it."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402

PEAKS = {"hbm_gbs": 6000.0, "fp64_flops": 1.25e12, "source": "measured"}
TWO = {"z_c2r": {"lines_per_transform": 2}, "z_r2c": {"lines_per_transform": 2}}
ONE = {"z_c2r": {"lines_per_transform": 1}, "z_r2c": {"lines_per_transform": 1}}


@pytest.mark.parametrize("name,desc,bound", [
    ("cross_z_r2c", TWO, "hbm"), ("curl_x_inverse6", TWO, "hbm"), ("fft_y_inverse", None, "hbm"),
    ("fft_z_c2r", TWO, "hbm"), ("fft_z_c2r", ONE, "alu"), ("fft_z_r2c", ONE, "alu"), ("update", TWO, "alu")])
@pytest.mark.parametrize("alu_frac", [0.97, 1.3])
def test_roof_follows_the_arithmetic(name, desc, bound, alu_frac):
    w = {"n": 256, "name": "none"}
    keep = bench.plain_keep((256, 256, 256))
    _, flops = bench.kernel_model(name, (256, 256, 256), "fp64", keep)
    ms = flops / (alu_frac * PEAKS["fp64_flops"]) * 1e3   # per launch
    roof, _ = bench.roofline_of([(name, 2, 2 * ms)], w, "fp64", 1, PEAKS, None, None, desc)
    assert roof["fp64_pipe_frac"] == pytest.approx(alu_frac)
    assert roof["bound"] == bound or (bound == "alu" and roof["frac"] > alu_frac)   # HBM nearer than the pipe
