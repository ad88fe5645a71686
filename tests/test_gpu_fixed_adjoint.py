"""The FP64 adjoint step in fixed point: cotangents of any size and zero ones, nodes outside
its range, every model, against the double-word adjoint (another code over populations).

Tolerance: the double-word form keeps about 47 bits an operation and its adjoint about 1e-11
relative over a few steps; a cotangent component may be 2^-4 of its node's largest, and
a gradient sums nine of them: 1e-9 of the largest gradient."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import flows
from paper_2602_21242_gb300.lattice import Lattice, run

pytestmark = pytest.mark.gpu


def _grads(prec, model, fields, cot, n, theta, tau):
    ny, nx = fields[0].shape
    with Lattice(nx, ny, theta, tau, model, prec) as lat:
        x = [torch.from_numpy(f).cuda().requires_grad_(True) for f in fields]
        out = run(lat, *x, n, 3)
        g = torch.autograd.grad(out, x, [torch.from_numpy(c).cuda() for c in cot])
        return np.stack([v.cpu().numpy() for v in g])


def _case(nx, ny, out_of_range):
    g = np.random.default_rng(nx)
    rho, ux, uy = flows.shear_wave(nx, ny, 0.1, 0.05)
    rho = rho + 0.02 * g.uniform(-1, 1, rho.shape)
    uy = uy + 0.05 * g.uniform(-1, 1, rho.shape)
    if out_of_range:
        rho[2:5, 3:9] = 5.0
        ux[7:9, 12:15] = 0.55
    cot = [g.standard_normal(rho.shape) for _ in range(3)]
    for c in cot:
        c[:, : nx // 2] = 0.0  # no cotangent reaches half of the nodes at first
    return (rho, ux, uy), cot


@pytest.mark.parametrize("model", [0, 1, 2, 3, 4])
@pytest.mark.parametrize("theta", [0.22, 1 / 3, 0.7])
@pytest.mark.parametrize("out_of_range", [False, True])
def test_against_the_double_word_adjoint(model, theta, out_of_range):
    fields, cot = _case(67, 22, out_of_range)
    a = _grads("f64", model, fields, cot, 4, theta, 0.9)
    b = _grads("f64df", model, fields, cot, 4, theta, 0.9)
    assert np.isfinite(a).all() and np.abs(a - b).max() <= 1e-9 * np.abs(b).max()


@pytest.mark.parametrize("k", [-900, -300, 40, 600])
def test_scaled_cotangents(k):
    """The derivative is linear, and a power of two goes through it exactly: bit for bit inside the
    exponents that the alignment takes, to rounding where the FP64 arithmetic takes over."""
    fields, cot = _case(40, 17, False)
    a = _grads("f64", 3, fields, cot, 5, 1 / 3, 0.7)
    b = _grads("f64", 3, fields, [np.ldexp(c, k) for c in cot], 5, 1 / 3, 0.7)
    b = np.ldexp(b, -k)
    if abs(k) < 700:
        assert np.array_equal(a, b)
    else:
        assert np.abs(a - b).max() <= 1e-12 * np.abs(a).max()
