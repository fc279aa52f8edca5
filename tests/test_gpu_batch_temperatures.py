"""The temperatures of a batch's models are those of its last run, whatever is read from the
grids in between: path-length tallies and their temperatures, temperatures of other counts
and another batch over the same grids. Copies and the same arithmetic: equality."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_species", [1, 2, 4])
def test_reads_of_the_grid_leave_the_batch_alone(n_species):
    nu = w.frequency_edges(20)
    sp = (w.two_species(nu) + [w.grey_species(20, 0.6, 0.4), w.grey_species(20, 0.2, 0.9)])
    grids = []
    for n_base in (4, 10):
        m = w.uniform_box_model(n_base, 20, 2.0, sp[:n_species])
        g = rt.Grid(m)
        g.emit_star(50_000)
        g.set_frozen_temperatures(frozen_field(m))
        g.transport(50_000, seed=9, mode=rt.REEMIT_FROZEN, estimators=rt.EST_PATHLENGTH)
        grids.append(g)
    kw = dict(mode=rt.REEMIT_FROZEN)
    a, b = rt.Batch(grids, [20_000, 50_000], seed=4, **kw), rt.Batch(grids, [9_000, 700], **kw)
    a.run()
    want = [g.temperatures() for g in grids]              # of the same counts
    assert all(np.array_equal(a.temperatures(i), T) for i, T in enumerate(want))
    for i, g in enumerate(grids):
        g.transport(50_000, seed=8, mode=rt.REEMIT_FROZEN, estimators=rt.EST_PATHLENGTH)
        assert g.pathlength().any()
        assert np.array_equal(a.temperatures(i), want[i])
        g.temperatures_pathlength()
        assert np.array_equal(a.temperatures(i), want[i])
        assert not np.array_equal(g.temperatures(), want[i])   # more packages
        assert np.array_equal(a.temperatures(i), want[i])
    b.run()
    for i, g in enumerate(grids):
        assert np.array_equal(b.temperatures(i), g.temperatures())
        assert np.array_equal(a.temperatures(i), want[i])
    # one grid twice in a batch: both see the sum of its counts, each in its own array
    twice = rt.Batch([grids[1], grids[1]], [5_000, 6_000], seed=4, **kw)
    twice.run_graph()
    T = grids[1].temperatures()
    assert np.array_equal(twice.temperatures(0), T) and np.array_equal(twice.temperatures(1), T)
    for x in (a, b, twice):
        x.close()
    for g in grids:
        g.close()
