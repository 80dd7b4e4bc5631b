"""The fixed-point entropy functions of the FP64 measure (fx64.cuh), compiled
for the host with g++ and checked against extended precision.  Bounds: the
units of the formats are 2^-63 (2^-z, log1p) and 2^-57 (u e^{-u^2/2}); a value
goes through at most a dozen truncations of one or two units, and the series
stop at terms below 1.5e-18, so 2^-58 = 3.5e-18 per function for the first two,
3.5e-18 + 1.1e-19 (the rounding of |u|) for log cosh, and 4 units of 2^-57 =
2.8e-17 for the product; FP64 itself carries 1.1e-16.  A sample that is not
finite must leave both sums not finite."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "c", "fx64_host", "fx64_check.cpp")
BOUNDS = {"exp": 3.5e-18, "log1p": 3.5e-18, "logcosh": 7e-18, "gauss": 2.8e-17}


def test_fixed_point_functions_against_extended_precision(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "fx64_check")
    # the CUDA declarations' stand-in is the one of the double-float check
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "tests", "c", "df64_host"),
                    "-I", os.path.join(ROOT, "paper_2409_05500_gb300", "csrc"),
                    SRC, "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    got = dict(line.split() for line in out.strip().splitlines())
    assert got.pop("nonfinite") == "1"
    assert set(got) == set(BOUNDS)
    for name, bound in BOUNDS.items():
        assert float(got[name]) <= bound, (name, got[name])
