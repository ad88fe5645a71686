"""Non-finite nodes met by fused diagnostics: the count in the error is the sum over all diagnosed steps of the nodes that
each met, in groups of every fill (below, at and above eight steps, and the call's end)."""
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import capi, flows
from paper_2602_21242_gb300.lattice import Lattice

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f64", "f64df", "f32", "f16"])
@pytest.mark.parametrize("calls,every", [((5,), 1), ((8,), 1), ((20,), 1), ((3, 1, 9), 1), ((25,), 3), ((4, 17), 2)])
def test_count_over_all_diagnosed_steps(prec, calls, every):
    nx, ny = 48, 40
    f = flows.random_populations(nx, ny, seed=1, spread=0.05)
    f[0, 20, 20] = np.nan
    with Lattice(nx, ny, 1 / 3, 0.6, "complete", prec) as lat:
        lat.set_state(torch.from_numpy(f).cuda())
        want = 0
        for t in range(sum(calls)):  # the nodes that the diagnosed step at time t meets
            if t % every == 0:
                want += int(lat.diagnostics(raise_nonfinite=False)[4])
            lat.step(1)
        lat.set_state(torch.from_numpy(f).cuda())
        lat.set_diagnostics_interval(every)
        for n in calls:
            lat.step(n)
        with pytest.raises(capi.LBMError) as e:
            lat.sync()
    got = int(re.search(r"(\d+) non-finite", str(e.value)).group(1))
    assert e.value.status == capi.LBM_ENONFINITE and got == want > 0


@pytest.mark.parametrize("prec", ["f64", "f64df"])
@pytest.mark.parametrize("value", [np.nan, -np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("every", [0, 1])
def test_nonfinite_populations_stay_so(prec, value, every):
    """A step hands a node's non-finite populations on as such (no finite stand-in), wherever they came from."""
    nx, ny = 48, 40
    f = flows.random_populations(nx, ny, seed=1, spread=0.05)
    f[[0, 1, 5], [20, 9, 30], [20, 40, 3]] = value
    with Lattice(nx, ny, 1 / 3, 0.6, "complete", prec) as lat:
        lat.set_diagnostics_interval(every)
        lat.set_state(torch.from_numpy(f).cuda())
        lat.step(1)
        got = lat.state().cpu().numpy()
    bad = ~np.isfinite(f).all(axis=0)
    for i, (cx, cy) in enumerate([(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]):
        assert np.array_equal(~np.isfinite(got[i]), np.roll(bad, (cy, cx), (0, 1))), i
