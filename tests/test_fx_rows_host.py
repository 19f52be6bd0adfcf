"""Fixed-point float64 operators row by row (CPU): the host packing and the
kernel's arithmetic (fx_pack.hpp, fx.hpp) compiled on the host. On inverses of
stiffness matrices with even, lognormal and jumping conductivities, and operands
that are dense, localised or spread over many decades, no row that is used in
fixed point may be further from its exact value, relative to sum |a_ij| |x_j|,
than the float64 sum."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_rows_are_as_accurate_as_float64(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    exe = str(tmp_path / "fx_rows_check")
    csrc = os.path.join(os.path.dirname(HERE), "paper_2410_14786_gb300", "csrc")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-I", csrc, os.path.join(HERE, "fx_rows_check.cpp"), "-o", exe,
                        "-lpthread"], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
