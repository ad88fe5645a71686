"""The default launch is more than its shape (several steps a launch on small lattices, the rows of diagnosed
FP64 steps, the rows of a small batch): reading the shape and setting it again changes nothing, and so does
choosing another one in between."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import capi, flows
from paper_2602_21242_gb300.batch import Batch
from paper_2602_21242_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def us_a_step(lat, steps=400, reps=15):
    best = float("inf")
    for _ in range(reps):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        lat.sync()
        e[0].record(lat.stream)
        lat.step(steps)
        e[1].record(lat.stream)
        lat.sync()
        best = min(best, 1e3 * e[0].elapsed_time(e[1]) / steps)
    return best


def tube(prec):
    """A tube of 800 nodes between two walls: with tiles 1.7 us a step, else two launches a step (4 and more)."""
    lat = Lattice(800, 1, 0.4, 0.6, "complete", prec)
    f = flows.random_populations(800, 1, seed=3, spread=0.02)
    lat.set_state(torch.from_numpy(f).cuda())
    return lat


def mask():
    m = np.zeros((1, 800), dtype=np.uint8)
    m[0, [0, 400, 799]] = 1
    return m


OTHER = {"f64": (0, 32, 4, 4), "f64df": (0, 32, 4, 4), "f32": (1, 0, 1, 4), "f16": (1, 0, 1, 4)}


@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16"])
@pytest.mark.parametrize("between", [False, True])
def test_setting_the_shape_that_was_read_is_the_default(prec, between):
    with tube(prec) as lat:
        lat.set_walls(mask())
        before = us_a_step(lat)
        shape = capi.lbm_get_launch_ex(lat.ctx)
        if between:
            capi.lbm_set_launch_ex(lat.ctx, *OTHER[prec])
        capi.lbm_set_launch_ex(lat.ctx, *shape)
        assert capi.lbm_get_launch_ex(lat.ctx) == shape
        assert us_a_step(lat) < 1.4 * before


@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16"])
def test_walls_set_under_another_shape(prec):
    """Walls that came while another shape was chosen act under the default shape as well."""
    got = {}
    for default_last in (False, True):
        with tube(prec) as lat:
            shape = capi.lbm_get_launch_ex(lat.ctx)
            capi.lbm_set_launch_ex(lat.ctx, *OTHER[prec])
            lat.set_walls(mask())
            if default_last:
                capi.lbm_set_launch_ex(lat.ctx, *shape)
            lat.step(41)
            got[default_last] = lat.state().cpu().numpy()
    assert np.array_equal(got[True], got[False])


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
@pytest.mark.parametrize("between", [False, True])
def test_batch_shape_that_was_read_is_the_default(prec, between):
    n = [24, 40, 61, 128]
    with Batch(n, n, [0.35] * 4, [0.7] * 4, "complete", prec) as b:
        launch = b.launch()
        if between:
            b.set_launch(0, 64, 4, 2)
        b.set_launch(*launch[:4])
        assert b.launch() == launch  # the shape and the tiles it comes to
