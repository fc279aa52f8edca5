"""A launch that its time budget ends leaves tallies that belong together: the packages counted
as escaped are those in the spectrum, one by one, in every walk and in a batch."""
import ctypes as C

import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RT_ERR_TIMEOUT = 4


def _counters(g):
    c = rt._Counters()
    code = rt.load().rt_get_counters(g._h, C.byref(c))
    return code, {k: int(getattr(c, k)) for k, _ in c._fields_}


def _check(g):
    sed = torch.zeros((2, g.n_dir, g.B), dtype=torch.int64, device="cuda")
    g.sed(out=sed)                        # a device read does not look at the status
    code, c = _counters(g)
    assert code == RT_ERR_TIMEOUT
    assert 0 < c["escaped"] < c["emitted"]
    assert int(sed[0].sum()) == c["escaped"]
    assert int(sed[1].sum()) <= c["escaped"] and c["errors"] == 0


def _grid(S, n):
    nu = w.frequency_edges(50)
    sp = (w.two_species(nu) + [w.grey_species(50, 0.6, 0.4), w.grey_species(50, 0.2, 0.9)])[:S]
    m = w.uniform_box_model(24, 50, 3.0, sp, max_level=1, refine=w.sphere_refine_fn(24, 0.3))
    g = rt.Grid(m)
    g.emit_star(n)
    g.set_frozen_temperatures(frozen_field(m))
    return g


@pytest.mark.parametrize("S,kw", [
    (1, {}), (2, {}), (2, dict(walk=rt.WALK_PATH)), (4, dict(walk=rt.WALK_LINKED)),
    (4, dict(walk=rt.WALK_PATH)), (2, dict(estimators=rt.EST_PATHLENGTH)),
    (2, dict(refill_period=4))])
def test_escaped_packages_are_in_the_spectrum(S, kw):
    n = 10 ** 8
    with _grid(S, n) as g:
        for seed in range(3):
            g.reset()
            g.transport(n, seed=seed, mode=rt.REEMIT_FROZEN, budget_s=0.002, **kw)
            _check(g)


def test_batch():
    n = 10 ** 8
    grids = [_grid(2, n) for _ in range(3)]
    b = rt.Batch(grids, [n] * 3, seed=1, mode=rt.REEMIT_FROZEN, budget_s=0.002)
    b.run()
    for g in grids:
        _check(g)
    b.close()
    for g in grids:
        g.close()
