"""Coefficients of the fixed-point collision, compiled for the host (tests/fixed_coefs_check.cpp): the nearest
integers of their formulas (113-bit arithmetic), the same on every machine, and cheap enough for a launch.

Bounds: correctly rounded is exact (at most half a unit). The host of a GPU prepares a launch in a few
microseconds, and these coefficients may take a tenth of that: 500 ns (measured 90 on Arm; software extended
precision took 670 there)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_21242_gb300", "csrc")


def _check(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "fixed_coefs_check")
    cmd = [cxx, "-O3", "-std=c++17", "-I", CSRC, os.path.join(HERE, "fixed_coefs_check.cpp"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    out = subprocess.run([exe, "20000", "3"], capture_output=True, text=True, check=True).stdout.split()
    return int(out[0]), float(out[1])


def test_coefficients_are_correctly_rounded(tmp_path):
    assert _check(tmp_path)[0] == 0


@pytest.mark.gpu
def test_coefficients_are_cheap_on_the_host_of_a_gpu(tmp_path):
    wrong, ns = _check(tmp_path)
    assert wrong == 0 and ns < 500.0, ns
