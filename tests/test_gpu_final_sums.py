"""The final sums of a call's last diagnosed steps run beside the steps that follow: a call of ten steps whose
first is diagnosed takes hardly longer than one without diagnostics, and its totals are those of that step.

Margin: 8 % (the sum beside the steps cost 4 %, after them 13 % and more)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import flows
from paper_2602_21242_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


def us_a_call(lat, steps, calls=20, reps=15):
    best = float("inf")
    for _ in range(reps):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        lat.sync()
        e[0].record(lat.stream)
        for _ in range(calls):
            lat.step(steps)
        e[1].record(lat.stream)
        lat.sync()
        best = min(best, 1e3 * e[0].elapsed_time(e[1]) / calls)
    return best


@pytest.mark.parametrize("n", [1024, 1448])
def test_one_diagnosed_step_a_call(n):
    with Lattice(n, n, 1 / 3, 0.6, "complete", "f16") as lat:
        lat.init(*(torch.from_numpy(a).cuda() for a in flows.shear_wave(n, n, U=0.1, amp=0.01)))
        plain = us_a_call(lat, 10)
        lat.set_diagnostics_interval(10)
        assert us_a_call(lat, 10) < 1.08 * plain


@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16"])
@pytest.mark.parametrize("nx,ny", [(64, 64), (500, 333)])
def test_totals_of_a_step_that_others_follow(prec, nx, ny):
    """Calls of one to three steps in turn, diagnosed every third step: the totals are those of the step, taken
    from lbm_diagnostics of the same state (FP64 sums; the fused ones of the shifted forms in FP32 within a block)."""
    tol = 1e-12 if prec.startswith("f64") else 64 * 2.0 ** -24
    f = flows.random_populations(nx, ny, seed=2, spread=0.05)
    with Lattice(nx, ny, 0.35, 0.8, "complete", prec) as ref, Lattice(nx, ny, 0.35, 0.8, "complete", prec) as lat:
        for x in (ref, lat):
            x.set_state(torch.from_numpy(f).cuda())
        lat.set_diagnostics_interval(3)
        t = 0
        for n in (1, 2, 3, 1, 3, 2, 3, 3):
            lat.step(n)
            t += n
            last = (t - 1) // 3 * 3
            if ref.time < last:
                ref.step(last - ref.time)
            got, when, _ = lat.step_diagnostics()
            want = np.array(ref.diagnostics())
            assert when == last
            assert np.abs(np.array(got)[:4] - want[:4]).max() <= tol * np.abs(f).sum()
