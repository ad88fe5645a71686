"""The fixed-point adjoint of one collision (lbm_fixed_adjoint.cuh), compiled for the host, against the transposed
Jacobian of the literal equations in extended precision (tests/fixed_adjoint_check.cpp).

Bounds, derived before the first run, in units of 2^-60 where the largest cotangent is below 2^56: a node takes about
85 products rounded by half a unit and as many sums and shifts that drop at most one, with weights of at most
4 (1 / theta, 1 / rho and k1 = 1 / (4 theta^2) below 6): 85 x 4 = 340 at the corners of the range. A relative
error of 1e-13 of the largest cotangent would be 3,600 units. Near equilibrium the error also stays below
that of the same derivative in binary64."""
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
    exe = str(tmp_path_factory.mktemp("fixed_adjoint") / "check")
    cmd = [cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I", CSRC, os.path.join(HERE, "fixed_adjoint_check.cpp"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return exe


@pytest.mark.parametrize("theta,tau", [(0.21, 0.501), (0.25, 3.0), (1 / 3, 0.515), (0.4, 0.55), (0.5, 1.0), (0.65, 0.6)])
def test_error_against_extended_precision(checker, theta, tau):
    out = subprocess.run([checker, "500", "5", repr(theta), repr(tau)], capture_output=True, text=True, check=True).stdout
    rows = [[float(x) for x in line.split()] for line in out.splitlines()]
    assert len(rows) == 15
    for model, family, n, taken, worst, rms, rms64 in rows:
        assert taken == n if family < 2 else taken > n // 10, (model, family, taken)
        assert worst <= 340.0, (model, family, worst)
        if family == 0:
            assert rms <= rms64, (model, rms, rms64)
