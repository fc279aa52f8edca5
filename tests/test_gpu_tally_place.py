"""Where a cell's path-length tally is kept (rows change places within blocks of 4096 leaves):
a thin beam along x adds the same length to the cells of its row and nothing to any other, on
grids that end before, at and after the end of a block, for every kernel and row length.

Tolerance: a tally is a sum of at most 1000 equal terms in FP32, 1000 x 2^-24 of it; the length
of a cell is the difference of two positions, 2^-20 of it."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("n_base", [3, 15, 16, 17, 33])
@pytest.mark.parametrize("kernel", [rt.KERNEL_POOL, rt.KERNEL_PLAIN_F32])
def test_tallies_lie_in_the_cells_crossed(S, n_base, kernel):
    nu = w.frequency_edges(16)
    sp = [w.grey_species(16, 0.1 * (k + 1), 0.0) for k in range(S)]
    tree = w.build_tree(n_base, 0)
    lo, hi = w.leaf_bounds_cm(tree, w.AU)
    ctr = (lo + hi) / 2
    rng = np.random.default_rng(n_base)
    row = ctr[rng.integers(tree.n_leaves), 1:]           # the beam's y and z
    on = np.abs(ctr[:, 1:] - row).max(axis=1) < 1e-6 * w.AU
    assert on.sum() == n_base
    rho = 1e-12 / w.AU * rng.uniform(1.0, 2.0, (S, tree.n_leaves))   # no package interacts
    star = w.Star(pos_cm=(-w.AU, *row), beam_dir=(1.0, 0.0, 0.0), kind=w.SOURCE_BEAM)
    m = w.explicit_model(tree, rho, 16, sp, star=star)
    n = 1000
    with rt.Grid(m) as g:
        g.emit_star(n)
        g.transport(n, seed=1, kernel=kernel, estimators=rt.EST_PATHLENGTH)
        tally = g.pathlength().astype(np.float64)
        T = g.temperatures_pathlength()
        g.reset()
        assert not g.pathlength().any()
    want = n * rho * np.array([s.kabs[0] for s in sp])[:, None] * (2 * w.AU / n_base)
    assert not tally[:, ~on].any() and not T[:, ~on].any() and (T[:, on] > 0).all()
    np.testing.assert_allclose(tally[:, on], want[:, on], rtol=1000 * 2.0 ** -24 + 2.0 ** -19)
