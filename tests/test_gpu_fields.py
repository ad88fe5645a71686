"""lbm_init, lbm_moments and lbm_diagnostics with sums and products in fixed point: fields on
both sides of the ranges that take it, against extended precision, and the batch's single
launch over all domains against single lattices.

Bounds. Initial populations: half an ulp of the storage type beyond 2^-50 (the FP64
arithmetic that the shifted forms reproduce makes at most four roundings of values below 4);
FP64 storage half an ulp and 24 units of 2^-60 below density 4, four roundings (2^-51 of
the density) elsewhere. Moments: the sum is exact (FP64 storage: populations truncated at
2^-60, nine of them) and rounded once; u = j (1/rho) adds three roundings."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import flows
from paper_2602_21242_gb300.batch import Batch
from paper_2602_21242_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu

C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
EPS = {"f64": 2.0 ** -53, "f64df": 2.0 ** -53, "f32": 2.0 ** -24, "f16": 2.0 ** -11}


def _fields(nx, ny, seed):
    g = np.random.default_rng(seed)
    rho = g.choice([1.0, 1.0, 1.0 + 1e-9, 0.7, 1.3, 1.99, 2.01, 3.9, 4.1, 0.01], (ny, nx)) * (1 + 1e-2 * g.uniform(-1, 1, (ny, nx)))
    rho[:3] = 1.0
    ux, uy = (g.choice([0.0, 1e-12, 1e-6, 1e-3, 0.1, 0.3, 0.4999999, 0.5, 0.6], (ny, nx)) * g.choice([-1, 1], (ny, nx))
              for _ in range(2))
    return rho, ux, uy


def _equilibrium(rho, ux, uy, theta):
    r, u, v, th = (np.asarray(a, dtype=np.longdouble) for a in (rho, ux, uy, theta))
    P = lambda a, w: 1 - th - w * w if a == 0 else (th + w * w + a * w) / 2
    return np.stack([r * P(a, u) * P(b, v) for a, b in C])


@pytest.mark.parametrize("theta", [0.15, 0.25, 1 / 3, 0.6])
@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16"])
def test_initial_populations(prec, theta):
    nx, ny = 133, 41
    rho, ux, uy = _fields(nx, ny, 3)
    with Lattice(nx, ny, theta, 0.8, "complete", prec) as lat:
        lat.init(*(torch.from_numpy(a).cuda() for a in (rho, ux, uy)))
        got = lat.state().cpu().numpy().astype(np.longdouble)
    want = _equilibrium(rho, ux, uy, theta)
    unit = np.longdouble(2) ** -60
    if prec in ("f64", "f64df"):
        bound = np.where((rho < 4)[None], np.abs(want) * 2 * EPS[prec] + 24 * unit, 0) + np.where(
            (np.maximum(np.abs(ux), np.abs(uy)) >= 0.5) | (rho >= 4) | (theta < 0.21), rho * 2.0 ** -51, 0)[None]
    else:
        rest = _equilibrium(1.0, 0.0, 0.0, theta)[:, None, None]
        bound = np.abs(want - rest) * 2 * EPS[prec] + 2.0 ** -50 * np.maximum(rho, 1)[None]
        if prec == "f16":
            bound = bound + 2.0 ** -25  # half the smallest half-precision step
    bound = bound + np.abs(want) * 2 * 2.0 ** -53  # state() adds the rest value in binary64
    assert (np.abs(got - want) <= bound).all(), float((np.abs(got - want) / bound).max())


@pytest.mark.parametrize("scale", [1.0, 0.05, 3.0])
def test_moments_and_diagnostics_f64(oracle, scale):
    nx, ny = 97, 70
    f = flows.random_populations(nx, ny, seed=4, spread=0.3) * scale
    g = np.random.default_rng(1)
    f[g.uniform(size=f.shape) < 0.02] *= -1.0
    f[:, 3, 5] *= 1e-7
    with Lattice(nx, ny, 0.3, 0.8) as lat:
        lat.set_state(torch.from_numpy(f).cuda())
        rho, ux, uy = (a.cpu().numpy() for a in lat.moments())
        diag = np.array(lat.diagnostics())
    e = f.astype(np.longdouble)
    j = [sum(c[k] * e[i] for i, c in enumerate(C)) for k in (0, 1)]
    r = e.sum(axis=0)
    mag = np.abs(f).sum(axis=0)
    sums = mag * 9 * 2.0 ** -53 + 9 * 2.0 ** -60  # FP64 sums outside the range, truncation inside
    assert (np.abs(rho - r) <= sums).all()
    for got, q in ((ux, j[0]), (uy, j[1])):
        want = q / r
        assert (np.abs(got - want) <= (sums * (1 + np.abs(want)) + np.abs(q) * 2.0 ** -51) / np.abs(r)).all()
    np.testing.assert_allclose(diag, oracle.diagnostics(f), rtol=1e-13, atol=1e-13 * scale * nx * ny)


@pytest.mark.parametrize("prec", ["f32", "f16"])
@pytest.mark.parametrize("size", [1.0, 1e-6, 1e-12])
def test_moments_of_small_deviations(prec, size):
    """Deviations of any size keep their relative accuracy (sums aligned to the largest)."""
    nx, ny, theta = 70, 33, 1 / 3
    w = np.array([(1 - theta if a == 0 else theta / 2) * (1 - theta if b == 0 else theta / 2) for a, b in C])
    if prec == "f16" and size < 1e-3:
        pytest.skip("below half precision")
    g = np.random.default_rng(9)
    # deviations exact in the storage type and in binary64 beside the rest value of 2^-k
    dev = g.integers(-1000, 1000, (9, ny, nx)) * 2.0 ** (-15 + round(np.log2(size)))
    f = w[:, None, None] + dev
    with Lattice(nx, ny, theta, 0.8, "complete", prec) as lat:
        lat.set_state(torch.from_numpy(f).cuda())
        stored = lat.state().cpu().numpy()
        rho, ux, uy = (a.cpu().numpy() for a in lat.moments())
    d = stored.astype(np.longdouble) - w[:, None, None]
    slack = 9 * 2.0 ** -53  # state() rounds each stored + rest value
    r = 1 + d.sum(axis=0)
    assert (np.abs(rho - r) <= slack + np.abs(r) * 2.0 ** -52).all()
    for got, k in ((ux, 0), (uy, 1)):
        q = sum(c[k] * d[i] for i, c in enumerate(C))
        assert (np.abs(got - q / r) <= (slack + np.abs(q) * 2.0 ** -50) / r).all()


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_batch_fields_equal_single_lattices(prec):
    sizes = [(64, 64), (1, 7), (33, 8), (90, 41), (5, 1), (128, 9)]
    nx, ny = zip(*sizes)
    theta, tau = [0.3, 1 / 3, 0.25, 0.4, 0.15, 0.35], [0.6, 0.8, 1.0, 0.7, 0.9, 0.55]
    fields = [_fields(a, b, 20 + k) for k, (a, b) in enumerate(sizes)]
    with Batch(nx, ny, theta, tau, "complete", prec) as b:
        for _ in range(2):  # twice: from either buffer
            b.init(*zip(*[[torch.from_numpy(a).cuda() for a in f] for f in fields]))
            states = [b.state(k).cpu().numpy() for k in range(len(sizes))]
            moments = [[m.cpu().numpy() for m in d] for d in b.moments()]
            b.step(1)
    for k, (a, c) in enumerate(sizes):
        with Lattice(a, c, theta[k], tau[k], "complete", prec) as lat:
            lat.init(*(torch.from_numpy(x).cuda() for x in fields[k]))
            assert np.array_equal(lat.state().cpu().numpy(), states[k])
            for got, want in zip(moments[k], lat.moments()):
                assert np.array_equal(got, want.cpu().numpy(), equal_nan=True)
