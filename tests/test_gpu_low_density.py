"""Densities in other units than 1 (0.6 down to 1e-37) in lbm_init, single lattices and batches, among
ordinary nodes: as accurate relative to the density as at density 1.

Tolerance: f^eq in binary64 takes at most four roundings of values of the density's size."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300.batch import Batch
from paper_2602_21242_gb300.lattice import Lattice
from test_gpu_fields import _equilibrium

pytestmark = pytest.mark.gpu

DENSITIES = [1.0, 0.6, 0.5, 0.49, 0.3, 1e-1, 1e-2, 1e-3, 1e-6, 1e-9, 1e-12, 1e-15, 1e-18, 1e-19, 1e-30, 1e-37]


def _fields(nx, ny, seed):
    g = np.random.default_rng(seed)
    rho = g.choice(DENSITIES, (ny, nx)) * (1 + 1e-2 * g.uniform(-1, 1, (ny, nx)))
    ux, uy = g.uniform(-0.4, 0.4, (2, ny, nx))
    return rho, ux, uy


def _gpu(fields):
    return [torch.from_numpy(a).cuda() for a in fields]


@pytest.mark.parametrize("prec", ["f64", "f64df"])
@pytest.mark.parametrize("theta", [1 / 3, 0.6])
def test_initial_populations(prec, theta):
    nx, ny = 133, 41
    fields = _fields(nx, ny, 1)
    with Lattice(nx, ny, theta, 0.8, "complete", prec) as lat:
        lat.init(*_gpu(fields))
        got = lat.state().cpu().numpy().astype(np.longdouble)
    assert (np.abs(got - _equilibrium(*fields, theta)) <= fields[0] * 2.0 ** -51).all()


def test_batch_initial_populations():
    sizes = [(64, 33), (5, 7), (120, 9)]
    fields = [_fields(nx, ny, k) for k, (nx, ny) in enumerate(sizes)]
    with Batch(*zip(*sizes), [0.35] * 3, [0.8] * 3, "complete", "f64") as b:
        b.init(*zip(*[_gpu(f) for f in fields]))
        for k, f in enumerate(fields):
            got = b.state(k).cpu().numpy().astype(np.longdouble)
            assert (np.abs(got - _equilibrium(*f, 0.35)) <= f[0] * 2.0 ** -51).all()
