"""A grid's arrays share allocations: the table rows kept with the tables or (past 4 MB)
apart, the walks' arrays inside or built later outside, tables built again after new dust.
The same counts each way, and all memory given back. Whole numbers: equality."""
import dataclasses

import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _model(S, level):
    nu = w.frequency_edges(100)
    sp = (w.two_species(nu) + [w.grey_species(100, 0.6, 0.4), w.grey_species(100, 0.2, 0.9)])[:S]
    return w.uniform_box_model(4, 100, 3.0, sp, max_level=level,
                               refine=w.sphere_refine_fn(4, 0.5) if level else None)


@pytest.mark.parametrize("S,level,n_temp", [(1, 0, 0), (2, 1, 5243), (2, 1, 5242), (4, 1, 0)])
def test_counts_and_memory(S, level, n_temp):   # 5242 rows of 100 bins: within 4 MB
    m = _model(S, level)
    T, n = frozen_field(m), 20_000

    def run(**kw):
        with rt.Grid(m, n_temp=n_temp) as g:
            g.emit_star(n)
            out = []
            for _ in range(2):      # the second time with tables built again
                g.set_frozen_temperatures(T)
                g.reset()
                g.transport(n, seed=3, mode=rt.REEMIT_FROZEN, **kw)
                out.append((g.counts(), g.sed()[0], g.temperatures()))
                kabs, ksca, gg = (np.ascontiguousarray(a[0]) for a in m.opacity_arrays())
                sp = m.species[0]
                assert rt.load().rt_set_dust(g._h, 0, kabs.ctypes.data, ksca.ctypes.data,
                                             gg.ctypes.data, g.B, int(sp.is_pah),
                                             int(sp.n_carbon)) == 0
            for a, b in zip(*out):
                assert np.array_equal(a, b)
            return out[0]

    ref = run(walk=rt.WALK_LINKED)
    for a, b in zip(ref, run(walk=rt.WALK_PATH)):
        assert np.array_equal(a, b)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(20):
        run(walk=rt.WALK_LINKED)
        run(walk=rt.WALK_PATH)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 4 << 20   # 40 grids of 1.5 to 20 MB
