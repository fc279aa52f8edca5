"""The pool's schedule -- packages parked and moved between lanes, interactions with full
warps, new packages for idle lanes -- changes no history: totals of counts, spectra and
counters against the replay of every package one by one (rt_trace: one thread each, no
pool), for package numbers around a warp's lanes and places, every batch size at its ends,
blocks of one to eight warps, capped histories, and a source outside the grid that some
packages miss it from. Equality for the walks that sum opacities as the replay does (one
and three species); those compiled for two or four sum them in another order, where a
history parts from the replay's once in 1e6 crossings at most: then a total may differ by
the largest histories of that many packages."""
import dataclasses

import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
COLUMNS = {"absorptions": 1, "scatters": 2, "crossings": 3, "escaped": 4, "capped": 5}


def _model(S, star):
    nu = w.frequency_edges(24)
    sp = (w.two_species(nu) + [w.grey_species(24, 0.6, 0.4, 0.3),
                               w.grey_species(24, 0.2, 0.9)])[:S]
    m = w.uniform_box_model(4, 24, 8.0, sp, max_level=2, refine=w.sphere_refine_fn(4, 0.5),
                            star=star)
    rng = np.random.default_rng(S)
    return dataclasses.replace(m, rho=m.rho * rng.choice([0.0, 0.4, 1.0, 3.0],
                                                         size=m.rho.shape[1])[None, :])


INSIDE = w.Star(pos_cm=(0.13 * w.AU, -0.21 * w.AU, 0.07 * w.AU))
OUTSIDE = w.Star(pos_cm=(0.2 * w.AU, 0.1 * w.AU, 1.0 * w.AU))   # on the upper boundary


@pytest.mark.parametrize("S,walk", [(1, "LINKED"), (2, "LINKED"), (2, "PATH"), (3, "PATH"),
                                    (4, "LINKED"), (4, "PATH")])
@pytest.mark.parametrize("star", ["inside", "outside"])
def test_every_schedule_gives_the_replayed_histories(S, walk, star):
    m = _model(S, INSIDE if star == "inside" else OUTSIDE)
    n_all = 40_000
    with rt.Grid(m) as g:
        g.emit_star(n_all)
        g.set_frozen_temperatures(frozen_field(m))
        runs = [(n, {}) for n in (1, 31, 32, 33, 63, 64, 65, 1000, n_all)]
        runs += [(n_all, kw) for kw in (
            dict(interaction_batch=1), dict(interaction_batch=2), dict(interaction_batch=32),
            dict(refill_period=1), dict(threads=32, blocks_per_sm=1),
            dict(threads=96, blocks_per_sm=2, interaction_batch=17), dict(max_events=3))]
        seen = {}
        for n, kw in runs:
            cap = kw.get("max_events", 0)
            if (n, cap) not in seen:
                seen[n, cap] = g.trace(np.arange(n), seed=5, max_events=cap)
            tr = seen[n, cap]
            g.reset()
            g.transport(n, seed=5, mode=rt.REEMIT_FROZEN, walk=getattr(rt, "WALK_" + walk), **kw)
            c, sed = g.counters(), g.sed()[0][0]
            assert c["errors"] == 0 and c["emitted"] == n
            assert c["absorptions"] == int(g.counts().sum())
            assert c["escaped"] + c["capped"] == n and int(sed.sum()) == c["escaped"]
            for name, col in COLUMNS.items():
                parted = 0 if S in (1, 3) else 2 + c["crossings"] // 10**6
                slack = parted * int(tr[:, col].max())
                assert abs(c[name] - int(tr[:, col].sum())) <= slack, (n, kw, name)


@pytest.mark.parametrize("S,bins,dirs,walk", [
    (1, 1024, 1, "LINKED"), (2, 1024, 1, "LINKED"), (6, 300, 1, "LINKED"), (6, 300, 1, "PATH"),
    (8, 1024, 3, "LINKED"), (3, 1024, 9, "PATH"), (3, 1024, 64, "LINKED")])
def test_tables_of_every_size_beside_the_places(S, bins, dirs, walk):
    # the places are part of the block's shared memory: launches whose tables alone stay
    # below 48 KB, or fill what the spectrum's choice of memory allows (200 KB)
    nu = w.frequency_edges(bins)
    sp = w.two_species(nu)[:S] + [w.grey_species(bins, 0.2 + 0.1 * s, 0.3)
                                  for s in range(max(S - 2, 0))]
    m = w.uniform_box_model(4, bins, 3.0, sp, max_level=1, refine=w.sphere_refine_fn(4, 0.5),
                            n_sed_dirs=dirs)
    n = 3000
    with rt.Grid(m) as g:
        g.emit_star(n)
        g.set_frozen_temperatures(frozen_field(m))
        tr = g.trace(np.arange(n), seed=8)
        for est in (0, rt.EST_PATHLENGTH):
            g.reset()
            g.transport(n, seed=8, mode=rt.REEMIT_FROZEN, walk=getattr(rt, "WALK_" + walk),
                        estimators=est)
            c, sed = g.counters(), g.sed()[0][0]
            assert c["errors"] == 0 and c["escaped"] == n == int(sed.sum())
            slack = 0 if S != 2 else 2 * int(tr[:, 1].max())
            assert abs(c["absorptions"] - int(tr[:, 1].sum())) <= slack
            assert c["absorptions"] == int(g.counts().sum())
