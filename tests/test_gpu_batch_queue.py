"""The batched launch hands every package of every model out exactly once, whatever a
warp takes at a time: in the frozen mode (histories independent of the schedule) its
counts, spectra and counters equal those of a launch per model."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
PACKAGES = [1, 31, 32, 33, 64, 65, 1000, 20_011, 7, 100_003]


@pytest.mark.parametrize("chunk,threads", [(0, 0), (1, 0), (32, 64), (33, 0), (100, 128),
                                           (5000, 0), (1 << 40, 0)])
def test_batch_equals_single_models(chunk, threads):
    models = [w.sphere_model(n_base=4 + 2 * (i % 3), n_bins=20 + i, tau_v=0.5 + i)
              for i in range(len(PACKAGES))]
    grids, single = [], []
    for i, (m, n) in enumerate(zip(models, PACKAGES)):
        g = rt.Grid(m)
        g.emit_star(n)
        g.set_frozen_temperatures(frozen_field(m))
        g.transport(n, seed=9 + i, mode=rt.REEMIT_FROZEN)
        single.append((g.counts(), g.sed()[0], g.counters()))
        grids.append(g)
    b = rt.Batch(grids, PACKAGES, seed=9, mode=rt.REEMIT_FROZEN, chunk=chunk, threads=threads)
    for _ in range(2):
        b.run()
        for g, (cnt, sed, c) in zip(grids, single):
            assert g.counters() == c
            assert np.array_equal(g.counts(), cnt)
            assert np.array_equal(g.sed()[0], sed)
    b.close()


def test_more_models_than_a_warp_scans_at_once():
    m = w.sphere_model(n_base=4, n_bins=16)
    T = frozen_field(m)
    grids = []
    for _ in range(67):
        g = rt.Grid(m)
        g.emit_star(500)
        g.set_frozen_temperatures(T)
        grids.append(g)
    npk = [500 if i % 5 else i % 3 for i in range(67)]
    b = rt.Batch(grids, npk, seed=1, mode=rt.REEMIT_FROZEN)
    b.run()
    assert [g.counters()["escaped"] for g in grids] == npk
    b.close()
