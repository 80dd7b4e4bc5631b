"""The sums of the fixed-point entropy functions (fx64.cuh), compiled for the host.
Bounds a sample, before any rounding to doubles: |w| is cut to units of 2^-57, so
|u| = |w| ln2 / 2 to 2.41e-18; log1p(2^-|w|) to 3.5e-18 for each of its two functions
and 2.4e-18 for the cut of its argument, 9.4e-18.  The conversion of a run of up to 200 samples: two units of 2^-52 of the
result, and absolutely the cut of the product with ln 2 (2^-57), the rounding of ln 2
(2^-64 a sample and a unit of |u|, at most 23 each) and the extended precision of the
check itself (2^-63 of a sum of |u| of at most 200 x 22.2 and of 200 ln 2, 5e-16):
1.2e-15; with a sample beyond the range, also one rounding of its |u| <= 127 in FP64,
2.9e-14."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "tests", "c", "fx64_host", "fx64_sums_check.cpp")
BOUNDS = {"abs": 2.41e-18, "log1p": 9.4e-18, "convert_logcosh": 1.2e-15,
          "convert_gauss": 1.2e-15, "beyond": 2.9e-14}


def test_fixed_point_sums_before_and_after_conversion(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "fx64_sums_check")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "tests", "c", "df64_host"),
                    "-I", os.path.join(ROOT, "paper_2409_05500_gb300", "csrc"),
                    SRC, "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    got = dict(line.split() for line in out.strip().splitlines())
    assert set(got) == set(BOUNDS)
    for name, bound in BOUNDS.items():
        assert float(got[name]) <= bound, (name, got[name])
