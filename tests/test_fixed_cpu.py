"""The fixed-point collision of the FP64 form (lbm_fixed.cuh), compiled for the host:
tests/fixed_check.cpp collides random nodes of every model (near equilibrium, random
populations, the corners of the accepted range, a fluid at rest) and compares them with
the literal equations in extended precision.

Bounds, derived before the first run: each stored population is rounded to binary64 once
(half an ulp); beyond that it is a sum of at most four moments, each of at most ten products
truncated by 1.25 units of 2^-60 with weights below one: 40 units (with rho < 4, |j| < 2).
The error also has to stay below that of the same equations in binary64, or (LBGK at
large tau, where hardly anything happens) within 1 % of the exact result's own rounding."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_21242_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path_factory.mktemp("fixed") / "fixed_check")
    cmd = [cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, os.path.join(HERE, "fixed_check.cpp"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return exe


def _rows(checker, n, theta, tau):
    out = subprocess.run([checker, str(n), "7", repr(theta), repr(tau)], capture_output=True, text=True, check=True)
    return [[float(v) for v in line.split()] for line in out.stdout.splitlines()]


@pytest.mark.parametrize("theta,tau", [(0.21, 0.501), (0.25, 3.0), (1 / 3, 0.515), (0.4, 0.55), (0.5, 1.0), (0.57, 50.0), (0.65, 0.6)])
def test_error_against_extended_precision(checker, theta, tau):
    rows = _rows(checker, 20_000, theta, tau)
    assert len(rows) == 24
    for model, family, n, taken, excess, rms, rms64, rounding in rows:
        assert taken == n if family in (0, 1, 3) else taken > n // 10, (model, family, taken)
        assert excess <= 40.0, (model, family, excess)
        assert rms <= max(rms64, 1.01 * rounding), (model, family, rms, rms64, rounding)


@pytest.mark.parametrize("theta,tau", [(0.2, 0.8), (0.66, 0.8), (1 / 3, 1e12)])
def test_coefficients_outside_the_range_are_left_out(checker, theta, tau):
    assert all(row[3] == 0 for row in _rows(checker, 100, theta, tau))
