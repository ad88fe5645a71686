"""Scratch of the fused diagnostics: at most four buffers of 40 bytes a block (the two groups of two that a
two-step launch needs) or a MiB, whatever shape is chosen, and the totals with groups of every size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import capi, flows
from paper_2602_21242_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def test_scratch_of_small_blocks_on_a_large_lattice():
    n = 4096
    blocks = (n // 64) * n  # blocks of 32 node pairs, one row each
    with Lattice(n, n, 1 / 3, 0.6, "complete", "f16") as lat:
        lat.sync()
        before = torch.cuda.mem_get_info()[0]
        capi.lbm_set_launch_ex(lat.ctx, 0, 32, 1, 1)
        used = before - torch.cuda.mem_get_info()[0]
        assert used <= 4 * 40 * blocks + (4 << 20), used


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("shape", [(0, 32, 1, 1), (0, 32, 1, 3), (0, 64, 2, 4)])
@pytest.mark.parametrize("every", [1, 2])
def test_totals_with_groups_of_every_size(prec, shape, every):
    """700 x 640 in blocks of one row (two steps a group) up to 8 x 64 nodes (eight)."""
    nx, ny, steps = 700, 640, 23
    f = flows.random_populations(nx, ny, seed=8, spread=0.05)
    last = (steps - 1) // every * every
    with Lattice(nx, ny, 0.35, 0.8, "complete", prec) as lat:
        capi.lbm_set_launch_ex(lat.ctx, *shape)
        lat.set_state(torch.from_numpy(f).cuda())
        lat.step(last)
        want = np.array(lat.diagnostics())
        lat.set_state(torch.from_numpy(f).cuda())
        lat.set_diagnostics_interval(every)
        lat.step(steps)
        got, when, _ = lat.step_diagnostics()
    tol = 1e-12 if prec == "f64" else 64 * 2.0 ** -24
    assert when == last and np.abs(np.array(got)[:4] - want[:4]).max() <= tol * np.abs(f).sum()
