"""The pool's walks on grids with an odd number of base cubes along an edge, where the mirrored
frame's coordinates are odd multiples of the base cube and the middle of the domain lies
inside a cell: linked and path walk give the same histories, and those of the plain FP32
kernel, which relocates the package from its base cube at every crossing.

Tolerance against the plain kernel: it steps an edge or corner and sums opacities in another
order; a history parts once in some 1e6 crossings at most and has fewer than 1e3 of them."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
N = 60_000


@pytest.mark.parametrize("S", [1, 2, 4])
@pytest.mark.parametrize("n_base,level", [(1, 0), (1, 4), (3, 0), (3, 2), (5, 4), (7, 1), (13, 3)])
def test_walks_agree(S, n_base, level):
    nu = w.frequency_edges(24)
    sp = (w.two_species(nu) + [w.grey_species(24, 0.6, 0.4, 0.3), w.grey_species(24, 0.2, 0.9)])[:S]
    even = w.uniform_box_model(2, 24, 2.0, sp)          # its density, on an odd grid
    tree = w.build_tree(n_base, level, w.sphere_refine_fn(n_base, 0.5))
    rng = np.random.default_rng(n_base)
    rho = even.rho[:, :1] * rng.choice([0.0, 0.3, 1.0, 2.5], size=tree.n_leaves)[None, :]
    m = w.explicit_model(tree, rho, 24, sp, star=w.Star(pos_cm=(0.13 * w.AU, -0.21 * w.AU, 0.0)))

    def run(g, **kw):
        g.reset()
        g.transport(N, seed=11, mode=rt.REEMIT_FROZEN, **kw)
        c = g.counters()
        assert c["errors"] == 0 and c["capped"] == 0 and c["emitted"] == c["escaped"] == N
        return g.counts().astype(np.int64), g.sed()[0].astype(np.int64)

    with rt.Grid(m) as g:
        g.emit_star(N)
        g.set_frozen_temperatures(frozen_field(m))
        cnt, sed = run(g, walk=rt.WALK_LINKED)
        path, sed_path = run(g, walk=rt.WALK_PATH)
        assert np.array_equal(path, cnt) and np.array_equal(sed_path, sed)
        for kw in (dict(kernel=rt.KERNEL_PLAIN_F32), dict(estimators=rt.EST_PATHLENGTH)):
            other, _ = run(g, **kw)
            assert np.abs(other - cnt).sum() <= 2e-3 * cnt.sum() + 20
