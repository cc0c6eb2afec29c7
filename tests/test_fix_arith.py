"""The fixed-point products and rotations of csrc/fft_fix.cuh, compiled for the
host, against exact 128-bit arithmetic: no operation has a mean error (a bias
adds up in phase over the lines of a transform), none is off by more than one and a
half units, and none overflows at the limit of its range.

Tolerances: an error lies within one unit either way, so its standard deviation is
below 0.6, and the mean of 400000 within 5 * 0.6 / sqrt(400000) = 0.005.  A single
operation rounds once by half a unit and drops products of low words below a unit."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def report(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    exe = str(tmp_path_factory.mktemp("fix") / "fix_arith")
    subprocess.run([nvcc, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I" + os.path.join(ROOT, "paper_1003_4322_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "fix_arith.cu"), "-o", exe], check=True, capture_output=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    return {name: (float(mean), float(worst)) for name, mean, worst in (line.split() for line in out.splitlines())}


@pytest.mark.parametrize("name,worst", [("cmul_w", 1.5), ("lrot", 1.5), ("half", 0.5)])
def test_no_bias(report, name, worst):
    assert report[name][0] < 0.005
    assert report[name][1] <= worst


def test_offset_of_input_0_reaches_every_output(report):
    assert report["offset"][0] == 0


def test_doubles_far_below_the_scale(report):
    assert report["from"][0] == 0
