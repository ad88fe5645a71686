"""FP64 storage, nodes outside the fixed-point range in bands of rows, so that a thread's column begins inside or
outside it and crosses the border several times: the same bits whatever rows a thread takes (one row, where no
row depends on another one's path, up to 32), and the totals of the diagnostics."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import capi, flows
from paper_2602_21242_gb300.lattice import Lattice
from test_gpu_launch_default import us_a_step

pytestmark = pytest.mark.gpu


def _state(nx, ny, kind):
    f = flows.random_populations(nx, ny, seed=11, spread=0.05)
    y, x = np.mgrid[:ny, :nx]
    if kind == "bands":  # whole warps: densities 0.3, 1, 6 by rows
        f *= np.choose((y // 5) % 3, [0.3, 1.0, 6.0])
    elif kind == "nodes":  # parts of warps as well
        f *= np.choose((y // 7 + x // 20) % 3, [1.0, 0.45, 5.0])
    else:  # everywhere
        f *= 9.0
    return f


@pytest.mark.parametrize("prec", ["f64", "f64df"])
@pytest.mark.parametrize("model", [0, 3, 5])
@pytest.mark.parametrize("kind", ["bands", "nodes", "all"])
@pytest.mark.parametrize("every", [0, 1])
def test_bits_do_not_depend_on_the_rows(prec, model, kind, every):
    nx, ny = 150, 97
    f, got = torch.from_numpy(_state(nx, ny, kind)).cuda(), {}
    for rows in (1, 2, 7, 32):
        with Lattice(nx, ny, 1 / 3, 0.9, model, prec) as lat:
            capi.lbm_set_launch_ex(lat.ctx, 0, 32, 2, rows)
            lat.set_diagnostics_interval(every)
            lat.set_state(f)
            lat.step(4)
            got[rows] = lat.state().cpu().numpy()
            if every:
                total = np.array(lat.step_diagnostics()[0])
                lat.set_state(f)
                lat.step(3)
                want = np.array(lat.diagnostics())
                assert np.abs(total[:4] - want[:4]).max() <= 1e-11 * float(f.abs().sum()) and total[4] == want[4] == 0
    assert np.isfinite(got[1]).all()
    for rows in (2, 7, 32):
        assert np.array_equal(got[rows], got[1]), rows


def test_time_of_a_flow_outside_the_range():
    """The double-word form's own arithmetic takes 1.3 times its fixed point; with every row tried in fixed point
    first the whole took 1.87 times, with the loop ended at such a row 1.65."""
    t = {}
    for rho in (1.0, 10.0):
        with Lattice(4096, 4096, 1 / 3, 0.8, "complete", "f64df") as lat:
            r, u, v = (torch.from_numpy(a).cuda() for a in flows.shear_wave(4096, 4096, U=0.1, amp=0.01))
            lat.init(rho * r, u, v)
            t[rho] = us_a_step(lat, steps=20)
    assert t[10.0] < 1.76 * t[1.0], t
