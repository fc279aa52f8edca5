"""Path-length tallies of every species count, whose rows are vectors of their own lengths: of
the pool, with images, and of a batch (models of equal and of mixed species counts), against
the plain FP32 kernel's, which adds species by species.

Tolerance: a history of the pool's parts from the plain kernel's once in some 1e6 crossings at
most (2e-3 of a total, as in the walks' test), and the FP32 sums of up to 1e5 increments in
another order differ by less."""
import ctypes as C

import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
N = 60_000


def _model(S):
    nu = w.frequency_edges(24)
    sp = (w.two_species(nu) + [w.grey_species(24, 0.15 * k, 0.4) for k in range(1, 7)])[:S]
    return w.uniform_box_model(6, 24, 2.0, sp, max_level=2, refine=w.sphere_refine_fn(6, 0.5),
                               star=w.Star(pos_cm=(0.13 * w.AU, -0.21 * w.AU, 0.07 * w.AU)))


def _grid(S):
    m = _model(S)
    g = rt.Grid(m)
    g.emit_star(N)
    g.set_frozen_temperatures(frozen_field(m))
    return g


def _plain(g, seed):
    g.reset()
    assert not g.pathlength().any()
    g.transport(N, seed=seed, mode=rt.REEMIT_FROZEN, kernel=rt.KERNEL_PLAIN_F32,
                estimators=rt.EST_PATHLENGTH)
    return g.pathlength().astype(np.float64), g.temperatures_pathlength()


def _close(tally, T, want, T_want):
    assert (tally > 0).any()
    for a, b in zip(tally.astype(np.float64), want):   # species by species
        assert np.abs(a - b).sum() <= 2e-3 * b.sum()
    assert np.array_equal(T > 0, tally > 0)
    assert np.abs(T - T_want).sum() <= 2e-3 * T_want.sum()


@pytest.mark.parametrize("S", range(1, 9))
def test_pool(S):
    with _grid(S) as g:
        g.transport(1, seed=0, mode=rt.REEMIT_FROZEN, estimators=rt.EST_PATHLENGTH)
        want, T_want = _plain(g, 11)
        g.reset()
        g.transport(N, seed=11, mode=rt.REEMIT_FROZEN, estimators=rt.EST_PATHLENGTH)
        _close(g.pathlength(), g.temperatures_pathlength(), want, T_want)
        g.reset()
        pob = np.full(24, -1, np.int32)
        pob[12] = 0
        g.set_images((0.0, 0.6, 0.8), pob, 9, 9, 1.05 * g.model.half_size)
        g.transport(N, seed=11, mode=rt.REEMIT_FROZEN, estimators=rt.EST_PATHLENGTH)
        _close(g.pathlength(), g.temperatures_pathlength(), want, T_want)


@pytest.mark.parametrize("species", [(1, 1), (2, 2), (3, 3), (4, 4), (8, 8), (5, 2, 4)])
def test_batch(species):
    grids = [_grid(S) for S in species]
    L = rt.load()
    arr = (C.c_void_p * len(grids))(*[g._h.value for g in grids])
    n = np.full(len(grids), N, dtype=np.uint64)
    o = rt._Opts(mode=rt.REEMIT_FROZEN, kernel=rt.KERNEL_POOL, estimators=rt.EST_PATHLENGTH)
    b = C.c_void_p()
    assert L.rt_batch_create(C.cast(arr, C.c_void_p), len(grids), n.ctypes.data, 7, C.byref(o), 0,
                             C.byref(b)) == 0
    assert L.rt_batch_run(b, 1, 1, None) == 0
    for i, g in enumerate(grids):
        tally, T = g.pathlength(), g.temperatures_pathlength()
        assert g.counters()["escaped"] == N
        want, T_want = _plain(g, 7 + i)                # seed + model
        _close(tally, T, want, T_want)
    L.rt_batch_destroy(b)
    for g in grids:
        g.close()
