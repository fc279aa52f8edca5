"""A batch's reset and temperatures, one launch each over all models: sizes from a few cells to
several blocks, odd numbers of counts, one, two, four and mixed species, the same grid twice;
against the single-model calls on the same tallies. The same arithmetic: equality."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu


def _grid(S, n_base, n):
    nu = w.frequency_edges(20)
    sp = (w.two_species(nu) + [w.grey_species(20, 0.6, 0.4), w.grey_species(20, 0.2, 0.9)])[:S]
    odd = n_base % 2          # 5^3 cells, the middle and its neighbour refined: 139
    m = w.uniform_box_model(n_base, 20, 2.0, sp, max_level=odd,
                            refine=lambda level, lo, hi: (lo[:, 0] >= 2) & (lo[:, 0] <= 3) &
                            (lo[:, 1] == 2) & (lo[:, 2] == 2)) if odd else \
        w.uniform_box_model(n_base, 20, 2.0, sp)
    g = rt.Grid(m)
    g.emit_star(n)
    g.set_frozen_temperatures(frozen_field(m))
    return g


@pytest.mark.parametrize("species", [(1, 1, 1), (2, 2, 2), (4, 4, 4), (1, 3, 2)])
def test_pass_equals_single_calls(species):
    grids = [_grid(S, n_base, 30_000) for S, n_base in zip(species, (2, 5, 20))]
    grids.append(grids[1])
    b = rt.Batch(grids[:3], [10_000, 20_000, 30_000], seed=4, mode=rt.REEMIT_FROZEN)
    first = None
    for run in (b.run, b.run_graph, b.run_graph):
        run()
        out = [(g.counts(), g.sed()[0], b.temperatures(i)) for i, g in enumerate(grids[:3])]
        clamped = [g.counters()["clamped"] for g in grids[:3]]
        for (c, s, T), g, k, n in zip(out, grids, clamped, (10_000, 20_000, 30_000)):
            assert int(s[0].sum()) == n        # one pass's packages, whatever came before
            assert np.array_equal(T, g.temperatures())
            assert g.counters()["clamped"] == 2 * k
        if first is not None:
            for x, y in zip(first, out):
                assert all(np.array_equal(p, q) for p, q in zip(x, y))
        first = out
    for g in grids[:3]:
        g.reset()
        assert not g.counts().any() and not g.sed()[0].any()
        assert not any(g.counters().values())
    twice = rt.Batch([grids[1], grids[3]], [5_000, 5_000], seed=4, mode=rt.REEMIT_FROZEN)
    twice.run()
    assert np.array_equal(twice.temperatures(0), twice.temperatures(1))
    assert int(grids[1].sed()[0][0].sum()) == 10_000
