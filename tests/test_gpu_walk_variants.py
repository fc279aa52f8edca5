"""The compiled forms of the pool's walk (species counts with vector rows, register
budgets, block sizes, the path-length tally) against each other and against the plain
FP32 kernel, which relocates the package from its base cube at every crossing, on grids
with cells of several levels, odd and even base counts, sources on corners, faces and
inside cells, and directions along the axes (a beam)."""
import dataclasses

import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
N = 120_000


def _model(S, n_base, level, star):
    nu = w.frequency_edges(24)
    sp = (w.two_species(nu) + [w.grey_species(24, 0.6, 0.4, 0.3), w.grey_species(24, 0.2, 0.9),
                               w.grey_species(24, 1.0)])[:S]
    m = w.uniform_box_model(2 * (n_base // 2), 24, 2.0, sp, max_level=level,
                            refine=w.sphere_refine_fn(n_base, 0.5), star=star)
    rng = np.random.default_rng(S)   # empty cells and a range of densities
    rho = m.rho * rng.choice([0.0, 0.3, 1.0, 2.5], size=m.rho.shape[1])[None, :]
    return dataclasses.replace(m, rho=rho)


STARS = {"corner": w.Star(), "inside": w.Star(pos_cm=(0.13 * w.AU, -0.21 * w.AU, 0.07 * w.AU)),
         "face": w.Star(pos_cm=(0.0, 0.31 * w.AU, -0.11 * w.AU)),
         "beam": w.Star(pos_cm=(-0.9 * w.AU, 0.11 * w.AU, 0.07 * w.AU), kind=w.SOURCE_BEAM,
                        beam_dir=(1.0, 0.0, 0.0)),
         "beam down": w.Star(pos_cm=(0.9 * w.AU, 0.0, 0.95 * w.AU), kind=w.SOURCE_BEAM,
                             beam_dir=(-0.6, 0.0, -0.8))}


def _run(g, **kw):
    g.reset()
    g.transport(N, seed=11, mode=rt.REEMIT_FROZEN, **kw)
    c = g.counters()
    assert c["errors"] == 0 and c["capped"] == 0 and c["emitted"] == c["escaped"] == N
    cnt = g.counts()
    assert int(cnt.sum()) == c["absorptions"]
    return cnt, g.sed()[0]


@pytest.mark.parametrize("S,n_base,level,star", [
    (1, 6, 2, "corner"), (2, 2, 4, "inside"), (2, 8, 0, "face"), (2, 6, 3, "beam"),
    (3, 4, 2, "beam down"), (4, 6, 2, "corner"), (4, 4, 4, "inside"), (4, 6, 1, "beam"),
    (5, 4, 1, "face")])
def test_variants_agree(S, n_base, level, star):
    m = _model(S, n_base, level, STARS[star])
    with rt.Grid(m) as g:
        g.emit_star(N)
        g.set_frozen_temperatures(frozen_field(m))
        ref, sed = _run(g, walk=rt.WALK_LINKED)
        # the same arithmetic whatever the register budget, block size, batch or refill
        for kw in (dict(blocks_per_sm=5), dict(threads=64), dict(threads=128, blocks_per_sm=2),
                   dict(interaction_batch=1, refill_period=7), dict(interaction_batch=32),
                   dict(walk=rt.WALK_PATH)):
            cnt, s = _run(g, **{"walk": rt.WALK_LINKED, **kw})
            assert np.array_equal(cnt, ref) and np.array_equal(s, sed), kw
        # the plain kernel steps an edge or corner and sums opacities in another order: a
        # history parts from the pool's once in some 1e6 crossings at most, and a history
        # has fewer than 1e3 of them
        cnt, s = _run(g, kernel=rt.KERNEL_PLAIN_F32)
        assert np.abs(cnt.astype(np.int64) - ref.astype(np.int64)).sum() <= 2e-3 * ref.sum() + 20
        # the tally changes nothing but rounding of the summed opacity, and sums the same
        # path lengths as the plain kernel's
        cnt, s = _run(g, walk=rt.WALK_LINKED, estimators=rt.EST_PATHLENGTH)
        assert np.abs(cnt.astype(np.int64) - ref.astype(np.int64)).sum() <= 2e-3 * ref.sum() + 20
        tally = g.pathlength()
        _run(g, kernel=rt.KERNEL_PLAIN_F32, estimators=rt.EST_PATHLENGTH)
        plain = g.pathlength()
        assert np.all(tally[m.rho == 0] == 0)
        np.testing.assert_allclose(tally.sum(axis=1), plain.sum(axis=1), rtol=2e-3)
