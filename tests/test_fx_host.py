"""Block fixed-point form of the float64 operators (CPU): fx.hpp compiled on
the host. Conversion and split over the whole range of float64, block sums at
their extreme values and at random against 128-bit integers, and whole dot
products (1 to 1500 terms) whose largest error must not exceed that of the
same products in float64."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fixed_point_form(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    exe = str(tmp_path / "fx_check")
    csrc = os.path.join(os.path.dirname(HERE), "paper_2410_14786_gb300", "csrc")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", csrc, os.path.join(HERE, "fx_check.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
