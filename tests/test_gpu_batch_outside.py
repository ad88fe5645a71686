"""FP64 batches with nodes outside the fixed-point range, more tiles than resident blocks and widths that leave
lanes without a column: persistent mode against graph mode, bit for bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import flows
from paper_2602_21242_gb300.batch import Batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["all", "bands", "nodes"])
@pytest.mark.parametrize("rows", [None, 1, 3, 16])
def test_persistent_equals_graph(kind, rows):
    n = [41, 200, 67, 99, 130, 33, 185, 1, 75, 31, 144, 160, 52, 193, 118, 70, 97, 129, 64, 177]
    ny = list(reversed(n))
    states = []
    for k, (a, b) in enumerate(zip(n, ny)):
        f = flows.random_populations(a, b, seed=k, spread=0.05)
        y, x = np.mgrid[:b, :a]
        f = f * (10.0 if kind == "all" else np.choose((y // 3) % 2, [1.0, 6.0]) if kind == "bands"
                 else np.choose((y // 5 + x // 9) % 3, [1.0, 0.4, 5.0]))
        states.append(torch.from_numpy(f).cuda())
    got = {}
    for mode in ("graph", "persistent"):
        with Batch(n, ny, [1 / 3] * 20, [0.8] * 20, "complete", "f64", mode=mode) as b:
            if rows is not None:
                b.set_launch(0, 64, 2, rows)
            for k, f in enumerate(states):
                b.set_state(k, f)
            b.step(5)
            b.sync()
            got[mode] = [b.state(k).cpu().numpy() for k in range(20)]
    for a, c in zip(got["graph"], got["persistent"]):
        assert np.isfinite(a).all() and np.array_equal(a, c)
