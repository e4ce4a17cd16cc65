"""The integer form of x^2 + y^2 rounded to FP64 (csrc/exact_sq.h, sq_sum_bits),
compiled for the host and compared bit for bit with the FPU."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_square_sum_bits(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    exe = tmp_path / "exact_sum_check"
    src = os.path.join(ROOT, "tests", "cpp", "exact_sum_check.cpp")
    inc = os.path.join(ROOT, "paper_2305_14398_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-I", inc, src, "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and "mismatches 0" in r.stdout, r.stdout + r.stderr
