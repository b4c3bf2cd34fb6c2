"""The logarithm of the scattered direct sums against the general-purpose
function that it replaces: at most 1 ulp everywhere.  Its error is half an ulp
of the result for the last sum, and an eighth each for the roundings of
r = m c - 1 and of the series where the table's rows meet the range around x = 1
that has c = 1 or 1/2 (there r is exact and the series off by 0.25 ulp)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_at_most_one_ulp(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "log_tab"
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", os.path.join(ROOT, "tests", "log_tab_harness.cpp"), "-o",
                    str(exe)], check=True)
    errors, special = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines()
    assert all(float(e) <= 1.0 for e in errors.split()), errors
    assert special.split() == ["1"] * 5
