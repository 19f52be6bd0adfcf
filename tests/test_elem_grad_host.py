"""Element term of the 3D adjoint gradient (CPU): elem_grad.hpp compiled on the
host. Where it takes its fixed-point form, the error relative to sum |K_ab| |u_a|
|lambda_b| may not exceed that of the float64 products."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


def test_fixed_point_where_it_is_accurate(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    exe = str(tmp_path / "elem_grad_check")
    csrc = os.path.join(os.path.dirname(HERE), "paper_2410_14786_gb300", "csrc")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I", csrc,
                        os.path.join(HERE, "elem_grad_check.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
