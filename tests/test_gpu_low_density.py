"""Densities in other units than 1 (0.6 down to 1e-37) in lbm_init, lbm_moments and
the adjoint's seed, single lattices and batches, among ordinary nodes: as accurate relative to the
density as at density 1.

Tolerances. f^eq in binary64 takes at most four roundings of values of the density's size. Moments:
eight additions of populations (u: of each sign) and, for u, the quotient's three roundings. The
gradient of no step at all is the identity: the seed's nine values and the sums over them take fewer than
64 roundings of terms of the size of g_rho + |g_u| / rho."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300.batch import Batch
from paper_2602_21242_gb300.lattice import Lattice, run
from test_gpu_fields import C, _equilibrium

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


def _check_moments(f, moments):
    e, mag = f.astype(np.longdouble), np.abs(f).sum(axis=0)
    r = e.sum(axis=0)
    rho, ux, uy = moments
    sums = mag * 9 * 2.0 ** -53
    assert (np.abs(rho - r) <= sums).all()
    for got, k in ((ux, 0), (uy, 1)):
        q = sum(c[k] * e[i] for i, c in enumerate(C))
        assert (np.abs(got - q / r) <= (sums * (1 + np.abs(q / r)) + np.abs(q) * 2.0 ** -51) / r).all()


@pytest.mark.parametrize("prec", ["f64", "f64df"])
def test_moments(prec):
    nx, ny = 133, 41
    with Lattice(nx, ny, 1 / 3, 0.8, "complete", prec) as lat:
        lat.init(*_gpu(_fields(nx, ny, 5)))
        _check_moments(lat.state().cpu().numpy(), [a.cpu().numpy() for a in lat.moments()])


def test_batch_moments():
    sizes = [(64, 33), (5, 7), (120, 9)]
    fields = [_fields(nx, ny, 10 + k) for k, (nx, ny) in enumerate(sizes)]
    with Batch(*zip(*sizes), [0.35] * 3, [0.8] * 3, "complete", "f64") as b:
        b.init(*zip(*[_gpu(f) for f in fields]))
        for k, m in enumerate(b.moments()):
            _check_moments(b.state(k).cpu().numpy(), [a.cpu().numpy() for a in m])


@pytest.mark.parametrize("prec", ["f64", "f64df"])
def test_gradient_of_no_step(prec):
    nx, ny = 70, 31
    fields = _fields(nx, ny, 6)
    g = np.random.default_rng(2)
    cot = g.uniform(-1, 1, (3, ny, nx))
    eps = 64 * (2.0 ** -53 if prec == "f64" else 2.0 ** -45)  # (double-word: its adjoint keeps about 47 bits)
    if prec == "f64df":
        fields[0][:] = np.maximum(fields[0], 1e-30)  # its exponents are FP32's: values below 1e-38 become zero
    with Lattice(nx, ny, 1 / 3, 0.8, "complete", prec) as lat:
        x = [a.requires_grad_(True) for a in _gpu(fields)]
        got = [v.cpu().numpy() for v in torch.autograd.grad(run(lat, *x, 0, 1), x, _gpu(cot))]
    rho, size = fields[0], np.abs(cot[0]) + (np.abs(cot[1]) + np.abs(cot[2])) / fields[0]
    assert (np.abs(got[0] - cot[0]) <= eps * size).all()
    for k in (1, 2):
        assert (np.abs(got[k] - cot[k]) <= eps * rho * size).all()
