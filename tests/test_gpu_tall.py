"""Lattices of more rows than two-row blocks have places for in a grid (131070): gradients in every form, against
the double-word adjoint, whose blocks have eight rows. Tolerance as between the two adjoints on other lattices: 1e-9 of the
largest gradient (FP32: 1e-4)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300.lattice import Lattice, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 131071), (3, 140001), (2, 300000)])
def test_gradients_of_tall_lattices(nx, ny):
    g = np.random.default_rng(ny)
    fields = [1.0 + 0.05 * g.uniform(-1, 1, (ny, nx)), *(0.05 * g.uniform(-1, 1, (2, ny, nx)))]
    cot = [torch.from_numpy(c).cuda() for c in g.standard_normal((3, ny, nx))]
    out = {}
    for prec in ("f64df", "f64", "f32"):
        with Lattice(nx, ny, 1 / 3, 0.8, "complete", prec) as lat:
            x = [torch.from_numpy(f).cuda().requires_grad_(True) for f in fields]
            out[prec] = torch.stack(torch.autograd.grad(run(lat, *x, 3, 2), x, cot)).cpu().numpy()
    want = out["f64df"]
    assert np.isfinite(want).all()
    for prec, tol in (("f64", 1e-9), ("f32", 1e-4)):
        assert np.abs(out[prec] - want).max() <= tol * np.abs(want).max(), prec
