"""Diagnosed steps: final sums of several steps a launch and the integer block reduction.

The totals after n steps diagnosed every k are those of the state before the last diagnosed step,
for counts below, at and above one group of final sums (8) and both groups (16), and lattices of one
block, of several rows a thread and with nodes outside the fixed-point range. The totals are sums of the
nodes' moments of f(x, t), taken here from get_state in extended precision.

Tolerance: each population is stored with a relative rounding of 2^-53 (FP64) and the totals are
rounded a few times on top; the fused sums use the step's own moments (FP32 forms: single precision
per node and block), so 2^-53 or 2^-24 times the sum of magnitudes times 64 bounds them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1], dtype=np.longdouble)
CY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1], dtype=np.longdouble)


@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16"])
@pytest.mark.parametrize("nx,ny", [(17, 1), (64, 64), (333, 150), (600, 517)])
@pytest.mark.parametrize("steps,every", [(1, 1), (8, 1), (9, 1), (17, 1), (34, 2), (50, 3)])
def test_last_diagnosed_totals(prec, nx, ny, steps, every):
    from paper_2602_21242_gb300.lattice import Lattice

    g = np.random.default_rng(nx * 7 + steps)
    rho = 1.0 + 0.02 * g.standard_normal((ny, nx))
    ux, uy = 0.05 * g.standard_normal((2, ny, nx))
    if prec == "f64" and nx > 17:
        rho[:, :5] *= 0.45  # below 1/2: nodes in floating point
    fields = [torch.from_numpy(a).cuda() for a in (rho, ux, uy)]
    last = (steps - 1) // every * every
    with Lattice(nx, ny, 1.0 / 3.0, 0.6, "complete", prec) as lat:
        lat.init(*fields)
        lat.step(last)
        f = lat.state().cpu().numpy().astype(np.longdouble).reshape(9, -1)
        lat.init(*fields)
        lat.set_diagnostics_interval(every)
        lat.step(steps)
        got, t, _ = lat.step_diagnostics()
    m0, jx, jy = f.sum(0), (CX[:, None] * f).sum(0), (CY[:, None] * f).sum(0)
    ke = 0.5 * (jx * jx + jy * jy) / m0
    eps = 2.0**-53 if prec.startswith("f64") else 2.0**-24
    assert t == last
    for k, (a, mag) in enumerate([(m0, np.abs(f).sum()), (jx, np.abs(f).sum()), (jy, np.abs(f).sum()),
                                  (ke, np.abs(f).sum())]):
        assert abs(float(got[k]) - float(a.sum())) <= 64 * eps * float(mag), (k, got[k], a.sum())


@pytest.mark.parametrize("steps", [5, 20])
def test_nonfinite_nodes_of_every_diagnosed_step_are_counted(steps):
    from paper_2602_21242_gb300 import capi
    from paper_2602_21242_gb300.lattice import Lattice

    with Lattice(48, 40, 1.0 / 3.0, 0.6, "complete", "f64") as lat:
        one = torch.ones((40, 48), dtype=torch.float64, device="cuda")
        lat.init(one, 0 * one, 0 * one)
        f = lat.state()
        f[0, 20, 20] = float("nan")
        lat.set_state(f)
        lat.set_diagnostics_interval(1)
        lat.step(steps)
        with pytest.raises(capi.LBMError):
            lat.step_diagnostics()
