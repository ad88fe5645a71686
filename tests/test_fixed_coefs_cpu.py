"""Coefficients of the fixed-point collision, compiled for the host (tests/fixed_coefs_check.cpp): the nearest
integers of their formulas (113-bit arithmetic), the same on every machine, and cheap enough for a launch.

Bounds: correctly rounded is exact (at most half a unit). The host prepares a launch in a few
microseconds, and these coefficients may take a tenth of that: 500 ns (measured 90 on Arm, 280 on x86; software
extended precision on Arm took 670)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_21242_gb300", "csrc")


def test_coefficients_are_correctly_rounded_and_cheap(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "fixed_coefs_check")
    cmd = [cxx, "-O3", "-std=c++17", "-I", CSRC, os.path.join(HERE, "fixed_coefs_check.cpp"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    out = subprocess.run([exe, "20000", "3"], capture_output=True, text=True, check=True).stdout.split()
    assert int(out[0]) == 0, out
    assert float(out[1]) < 500.0, out
