"""Batches around and beyond the 256 models that a warp weighs together: every package of every
model is handed out once, whatever the models' shares (equal, most of them empty, one large
among small ones at either end, none at all), and counts and spectra are those of a launch per
model (frozen mode: the schedule changes no history)."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu


def _plans(n):
    i = np.arange(n)
    return {"equal": np.full(n, 40), "ragged": i * 37 % 101, "sparse": np.where(i % 61, 0, 700),
            "large first": np.where(i, 20, 50_000), "large last": np.where(i < n - 1, 20, 50_000),
            "one": np.where(i == n // 2, 1, 0), "none": np.zeros(n, int)}


@pytest.mark.parametrize("n,threads", [(255, 0), (256, 0), (257, 64), (600, 0), (1100, 128)])
def test_every_package_once(n, threads):
    m = w.sphere_model(n_base=4, n_bins=16)
    T = frozen_field(m)
    grids = []
    for _ in range(n):
        g = rt.Grid(m)
        g.emit_star(50_000)
        g.set_frozen_temperatures(T)
        grids.append(g)
    alone = rt.Grid(m)
    alone.emit_star(50_000)
    alone.set_frozen_temperatures(T)
    for name, plan in _plans(n).items():
        b = rt.Batch(grids, plan, seed=3, mode=rt.REEMIT_FROZEN, threads=threads)
        for _ in range(2):
            b.run(temperatures=False)
            c = [g.counters() for g in grids]
            assert [x["emitted"] for x in c] == list(plan), name
            assert [x["escaped"] for x in c] == list(plan), name
        b.close()
        for i in (0, n // 2, n - 1):
            alone.reset()
            alone.transport(int(plan[i]), seed=3 + i, mode=rt.REEMIT_FROZEN)
            assert np.array_equal(alone.counts(), grids[i].counts())
            assert np.array_equal(alone.sed()[0], grids[i].sed()[0])
    for g in grids + [alone]:
        g.close()
