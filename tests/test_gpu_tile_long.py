"""Several steps a launch on long, thin lattices (regions of more than 1024 columns, the sizes where an
inexact row index would show) against single steps of the same form, bit for bit."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_2602_21242_gb300 import flows
from test_gpu_tile import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,nx,ny", [("f64", 160533, 1), ("f64df", 180001, 1), ("f32", 320000, 1),
                                        ("f32", 400001, 1), ("f16", 300000, 2), ("f16", 640003, 1), ("f16", 130001, 7)])
@pytest.mark.parametrize("walls", [False, True])
def test_long_lattices_equal_single_steps(prec, nx, ny, walls):
    f0 = flows.random_populations(nx, ny, seed=nx, spread=0.1)
    mask = np.random.default_rng(nx).uniform(size=(ny, nx)) < 0.05 if walls else None
    args = (f0, 0.35, 0.8, 3, prec, (41, 2), 0, mask)
    got, _ = _run(*args, False)
    want, _ = _run(*args, True)
    assert np.isfinite(want).all() and np.array_equal(got, want)
