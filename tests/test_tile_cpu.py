"""Index arithmetic of the several-steps-a-launch tiles (lbm_tile.h), compiled for the host:
tests/tile_check.cu takes every plan that tile_plan makes for lattices from a few columns to
10^6 with 1 to 100 rows, and compares the row of every index of every region with integer
division. Exact: no wrong index."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2602_21242_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no CUDA compiler")
    exe = str(tmp_path_factory.mktemp("tile") / "tile_check")
    cmd = [nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC,
           "-I", os.path.join(os.path.dirname(HERE), "include"), os.path.join(HERE, "tile_check.cu"), "-o", exe]
    res = subprocess.run(cmd, capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return exe


def _run(checker, *args):
    out = subprocess.run([checker, *map(str, args)], capture_output=True, text=True, check=True).stdout
    return [int(v) for v in out.split()]  # widths, planned, largest region, wrong indices, dear plans


@pytest.mark.parametrize("nx,ny,planned", [(378, 413, 0), (391, 383, 0), (450, 450, 0), (2042, 106, 0), (256, 256, 1),
                                           (512, 512, 1), (984, 105, 1), (5000, 31, 1), (284, 670, 1)])
def test_fp16_line_to_single_steps(checker, nx, ny, planned):
    """FP16 single steps that are one wave of CTAs are faster than tiles from about 150,000 nodes (measured: 3.3 to
    3.6 us a step against 3.8 to 4.3); below, and where they take two waves, the tiles are."""
    assert _run(checker, 2, 0, 152, ny, nx, nx, 1)[1] == planned


@pytest.mark.parametrize("prec", [0, 1, 2, 3])
@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("ny", [1, 2, 3, 4, 5, 7, 20, 100])
def test_rows_of_every_planned_region(checker, prec, walls, ny):
    # odd strides, so that ragged tiles of every size come up; wider lattices take no plan
    plans = 0
    for sms, lo, hi, stride in [(152, 1, 10_000 // ny, 37), (152, 10_000 // ny, 1_000_000 // ny, 4999 // ny * 2 + 1),
                                (148, 10_000 // ny, 1_000_000 // ny, 9973 // ny * 2 + 1), (20, 1, 100_000 // ny, 997),
                                (1, 1, 5000, 61)]:
        widths, planned, largest, wrong, dear = _run(checker, prec, walls, sms, ny, max(lo, 1), hi, stride)
        assert wrong == 0 and dear == 0, (sms, lo, hi, largest)
        plans += planned
    assert plans > 0
