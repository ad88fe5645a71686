"""Tuning never leaves a lattice or a batch slower than its default launch: the default is among what the tuner
times, and an entry of the cache that names it brings it back on lattices of the same class.

Margin: 15 %, a multiple of what two timings of one launch differ by; without the default these cases lost 25 %
and more."""
import json

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2602_21242_gb300 import capi, flows, tune
from paper_2602_21242_gb300.batch import Batch
from paper_2602_21242_gb300.lattice import Lattice
from test_gpu_launch_default import mask, us_a_step

pytestmark = pytest.mark.gpu


def _lattice(nx, ny, prec, walls):
    lat = Lattice(nx, ny, 1 / 3, 0.6, "complete", prec)
    lat.init(*(torch.from_numpy(a).cuda() for a in flows.shear_wave(nx, ny, U=0.1, amp=0.01)))
    if walls:
        lat.set_walls(mask())
    return lat


@pytest.mark.parametrize("nx,ny,prec,walls", [(64, 64, "f64", False), (800, 1, "f64", True), (800, 1, "f32", True),
                                              (512, 512, "f32", False)])
def test_tuned_lattice_is_not_slower(tmp_path, nx, ny, prec, walls):
    path = str(tmp_path / "tune.json")
    with _lattice(nx, ny, prec, walls) as lat:
        before = us_a_step(lat)
        _, ms = tune.tune_lattice(lat, path=path)
        assert ms > 0 and us_a_step(lat) < 1.15 * before
    with _lattice(nx, ny, prec, walls) as lat:  # from the cache, after another shape
        shape = (0, 32, 4, 4)
        capi.lbm_set_launch_ex(lat.ctx, *shape)
        _, ms = tune.tune_lattice(lat, path=path)
        assert ms is None and us_a_step(lat) < 1.15 * before


def test_cached_default_holds_for_the_size_class(tmp_path):
    path = str(tmp_path / "tune.json")
    with _lattice(64, 64, "f64", False) as lat:
        tune.tune_lattice(lat, path=path)
    with _lattice(64, 60, "f64", False) as lat:
        before = us_a_step(lat)
        assert tune.tune_lattice(lat, path=path)[1] is None
        assert us_a_step(lat) < 1.15 * before


def test_entries_chosen_without_the_default_are_not_used(tmp_path):
    path = str(tmp_path / "tune.json")
    with _lattice(64, 64, "f64", False) as lat:
        gpu = torch.cuda.get_device_name().replace(" ", "_")
        tune._store(path, f"{gpu}|lattice|2^12|nx=64|prec{lat.prec}|model{lat.model}", {"shape": [0, 32, 8, 32], "ms_per_step": 1.0})
        assert tune.tune_lattice(lat, path=path)[1] is not None
    assert len(json.load(open(path))) == 2


@pytest.mark.parametrize("prec", ["f64", "f32", "f16"])
def test_tuned_batch_is_not_slower(tmp_path, prec):
    path = str(tmp_path / "tune.json")
    n = [24, 40, 61, 128]
    fields = list(zip(*[[torch.from_numpy(a).cuda() for a in flows.shear_wave(k, k, U=0.1, amp=0.01)] for k in n]))

    def batch():
        b = Batch(n, n, [0.35] * 4, [0.7] * 4, "complete", prec)
        b.init(*fields)
        b.step(400)
        return b

    with batch() as b:
        before = us_a_step(b)
        assert tune.tune_batch(b, path=path)[1] > 0
        b.step(400)
        assert us_a_step(b) < 1.15 * before
    with batch() as b:
        b.set_launch(0, 64, 4, 2)
        assert tune.tune_batch(b, path=path)[1] is None
        b.step(400)
        assert us_a_step(b) < 1.15 * before
