"""Warp votes in routines that lanes may leave at different times (columns beyond a lattice's edge, ragged rows): a
mask of active lanes is used where it is taken, never kept over a loop, where it could hold lanes that have left and
the vote would wait for them for ever; and a kernel that goes through several tiles brings its warps together
after each."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_21242_gb300", "csrc")


def test_no_mask_of_active_lanes_is_kept():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        for line in open(path):
            code = line.split("//")[0]
            assert not re.search(r"=\s*__activemask\(\)", code), (os.path.basename(path), line.strip())
            assert not re.search(r"__syncwarp\(\s*[a-z_]", code), (os.path.basename(path), line.strip())


def test_warps_meet_after_each_tile_of_the_persistent_batch_kernel():
    text = open(os.path.join(CSRC, "lbm_batch_kernels.cuh")).read()
    body = text[text.index("batch_persistent_kernel("):]
    loop = body[body.index("for (int t = blockIdx.x"): body.index("grid_sync(")]
    assert loop.index("update_tile<") < loop.index("__syncwarp();")
