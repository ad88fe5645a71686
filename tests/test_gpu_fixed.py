"""The FP64 form's choice between the fixed-point and the floating-point collision: nodes
on both sides of every limit of the range (density, velocity, population sign and size,
temperature) in one lattice, one step against the oracle, and bit for bit the same under
launches that put different nodes into a warp.

Tolerance: the floating-point collision chains about a hundred binary64 operations whose
errors 1/(4 theta^2) <= 11 amplifies: 100 x 11 x 2^-53 = 1.2e-13 of the node's scale, its
largest population times the amplification of the populations' rounding in u = j/rho
(sum |f| / |rho|) and of u in the products' sixth powers (rho u^2 in N times P C^2).
Nodes beyond |u| = 2 (a density that cancels) are compared between launches only."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import capi, flows
from paper_2602_21242_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def _state(oracle, nx, ny, theta, seed):
    g = np.random.default_rng(seed)
    rho = g.choice([0.3, 0.499, 0.5, 0.501, 1.0, 1.5, 3.99, 4.0, 4.01, 40.0], (ny, nx)) * (1 + 1e-3 * g.uniform(-1, 1, (ny, nx)))
    ux, uy = (g.choice([0.0, 1e-9, 0.1, 0.49, 0.499999, 0.5, 0.51, -0.3, -0.5001], (ny, nx)) for _ in range(2))
    rho[:, : nx // 2], ux[:, : nx // 2], uy[:, : nx // 2] = 1.0, 0.1, -0.05  # half of it well inside
    # the pulled populations of a node: its own equilibrium, disturbed, a few negated or zero
    f = oracle.init(rho, ux, uy, theta)
    f = f * (1 + g.choice([0.0, 1e-3, 0.3], (1, ny, nx)) * g.uniform(-1, 1, f.shape))
    f[g.uniform(size=f.shape) < 0.01] *= -1.0
    f[g.uniform(size=f.shape) < 0.01] = 0.0
    return np.ascontiguousarray(f)


@pytest.mark.parametrize("theta", [0.15, 0.21, 1 / 3, 0.65, 0.7])
@pytest.mark.parametrize("model", [0, 1, 2, 3, 4, 5])
def test_both_paths_of_one_step(oracle, model, theta):
    nx, ny, tau = 150, 37, 0.77
    f = _state(oracle, nx, ny, theta, 3 + model)
    f[:, 5, 7] = np.nan
    f[3, 20, 100] = np.inf
    ref = oracle.run(f, theta, tau, model, 1)
    out = []
    for launch in ((0, 64, 2, 32), (0, 32, 1, 64), (0, 96, 1, 1), (1, 0, 1, 5)):
        with Lattice(nx, ny, theta, tau, model) as lat:
            capi.lbm_set_launch_ex(lat.ctx, *launch)
            lat.set_diagnostics_interval(1)
            lat.set_state(torch.from_numpy(f).cuda())
            lat.step(1)
            out.append(lat.state().cpu().numpy())
            diag = lat.step_diagnostics(raise_nonfinite=False)
            assert diag[0][4] == 2
    for got in out[1:]:
        same = (got == out[0]) | (np.isnan(got) & np.isnan(out[0]))
        assert same.all()
    finite = np.isfinite(ref)
    assert np.array_equal(finite, np.isfinite(out[0]))
    with np.errstate(invalid="ignore", divide="ignore"):
        rho, ux, uy = oracle.moments(f)
        scale = np.abs(f).max(axis=0) * np.abs(f).sum(axis=0) / np.abs(rho) * (1 + np.abs(ux) + np.abs(uy)) ** 6
        scale[~(np.maximum(np.abs(ux), np.abs(uy)) < 2.0)] = np.inf
    scale = np.stack([np.roll(scale, (b, a), (0, 1)) for a, b in
                      ((0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1))])
    err = np.abs(out[0] - ref)[finite] / scale[finite]
    assert err.max() <= 1.2e-13, err.max()


def test_diagnostics_of_both_paths(oracle):
    """Fused sums over nodes of both paths (exact integer sums and FP64 sums) against the state's."""
    nx, ny, theta, tau = 130, 70, 0.3, 0.8
    f = _state(oracle, nx, ny, theta, 11)
    with Lattice(nx, ny, theta, tau) as lat:
        lat.set_diagnostics_interval(1)
        lat.set_state(torch.from_numpy(f).cuda())
        lat.step(1)
        got = np.array(lat.step_diagnostics()[0])
    np.testing.assert_allclose(got, oracle.diagnostics(f), rtol=1e-13, atol=1e-11)
