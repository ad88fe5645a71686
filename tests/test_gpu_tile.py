"""Several steps a launch on small lattices (the default there) against single steps of the
same form, bit for bit: sizes that leave ragged tiles, that one tile spans in x, in y or in
both, odd step counts, diagnosed steps in between, walls, and nodes outside the FP64
form's fixed-point range. The single steps are those of a chosen launch shape
(lbm_set_launch_ex), which switches the several-step tiles off."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import capi, flows
from paper_2602_21242_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def _run(f0, theta, tau, model, prec, steps, every, mask, single):
    _, ny, nx = f0.shape
    with Lattice(nx, ny, theta, tau, model, prec) as lat:
        if single:
            kind = 0 if prec in ("f64", "f64df") or nx < 32 else 1
            capi.lbm_set_launch_ex(lat.ctx, kind, *((32, 4, 4) if kind == 0 else (0, 1, 4)))
        lat.set_walls(mask)
        lat.set_diagnostics_interval(every)
        lat.set_state(torch.from_numpy(f0).cuda())
        diags = []
        for n in steps:
            lat.step(n)
            diags.append(lat.step_diagnostics()[0] if every else lat.diagnostics())
        return lat.state().cpu().numpy(), np.array(diags)


@pytest.mark.parametrize("nx,ny", [(1, 1), (2, 3), (1, 200), (800, 1), (64, 64), (61, 47), (130, 3), (34, 96), (2, 500)])
@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16"])
@pytest.mark.parametrize("every,walls", [(0, False), (7, False), (5, True)])
def test_tiles_equal_single_steps(nx, ny, prec, every, walls):
    if prec in ("f32", "f16") and nx < 32 and nx % 2:
        pytest.skip("single nodes there: no tiles")
    f0 = flows.random_populations(nx, ny, seed=nx + 3 * ny, spread=0.1)
    mask = None
    if walls:
        mask = np.random.default_rng(nx).uniform(size=(ny, nx)) < 0.15
    for model in (0, 1, 3) if (nx, ny) == (61, 47) else (3,):
        args = (f0, 0.35, 0.8, model, prec, (1, 23, 40, 2), every, mask)
        got, dg = _run(*args, False)
        want, dw = _run(*args, True)
        assert np.array_equal(got, want), (model, np.abs(got - want).max())
        # sums: FP64 storage exact or FP64; the shifted forms in FP32 within a block (at most 60 roundings)
        tol = 1e-12 if prec in ("f64", "f64df") else 60 * 2.0 ** -24
        scale = np.abs(f0).sum()
        assert np.abs(dg[:, :4] - dw[:, :4]).max() <= tol * scale and np.array_equal(dg[:, 4], dw[:, 4])


@pytest.mark.parametrize("model", [0, 3, 5])
@pytest.mark.parametrize("prec", ["f64", "f64df"])
def test_nodes_outside_the_fixed_point_range(model, prec):
    """A dense spot (density 6) and a fast one among ordinary nodes."""
    nx, ny, theta = 48, 40, 1 / 3
    f0 = flows.random_populations(nx, ny, seed=5, spread=0.05)
    f0[:, 10:14, 10:14] *= 6.0
    f0[1, 30:33, 5:9] += 0.8
    got, _ = _run(f0, theta, 0.9, model, prec, (9,), 0, None, False)
    want, _ = _run(f0, theta, 0.9, model, prec, (9,), 0, None, True)
    assert np.isfinite(want).all() and np.array_equal(got, want)
