"""Kernels launched with programmatic serialization may be resident while the grid before them still
writes what they read: those that load through ordinary C++ pointers take them without
__restrict__ (which would let the compiler turn the loads into read-only ones or move them
above the wait for that grid), and every one of them waits."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2602_21242_gb300", "csrc")


@pytest.mark.parametrize("file,kernel", [("lbm_kernels.cuh", "step_kernel_f64"), ("lbm_kernels.cuh", "step_kernel_f64_float"),
                                         ("lbm_kernels.cuh", "step_kernel_df"), ("lbm_tile.cuh", "tile_steps_kernel"),
                                         ("lbm_adjoint.cu", "adj_step_f64_kernel"), ("lbm_adjoint.cu", "adj_step_pair_kernel")])
def test_sources_of_overlapping_kernels_are_not_restrict(file, kernel):
    text = open(os.path.join(CSRC, file)).read()
    m = re.search(r"\b%s\(\s*const [^{]*?\)\s*\{" % kernel, text)
    assert m, kernel
    for p in m.group(0).split(","):
        if "*" in p and "partials" not in p and "walls" not in p:
            assert "__restrict__" not in p, (kernel, p.strip())


@pytest.mark.parametrize("file,kernel,first", [("lbm_tile.cuh", "tile_steps_kernel", "base[i * plane"),
                                               ("lbm_adjoint.cu", "adj_step_f64_kernel", "adj_load_f64(f"),
                                               ("lbm_adjoint.cu", "adj_step_pair_kernel", "pair_plain(q")])
def test_the_kernels_wait_before_they_load(file, kernel, first):
    text = open(os.path.join(CSRC, file)).read()
    body = text[text.index(kernel + "(const"):]
    assert 0 < body.index("pdl_wait();") < body.index(first)
