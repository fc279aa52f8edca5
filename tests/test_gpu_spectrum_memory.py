"""The escaped spectrum in shared or in global memory: it is in shared memory only where it
costs no resident block. Sizes on both sides of that line (one block per SM always leaves room
for it, the launch's own choice of blocks does not), every walk, with images and with the
path-length tally: the same spectra, counts and counters, and the packages they should hold."""
import math

import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bins,dirs", [(64, 1), (200, 8), (257, 8), (333, 8), (1024, 1), (1024, 9)])
@pytest.mark.parametrize("S,kw", [
    (1, {}), (2, {}), (2, dict(walk=rt.WALK_PATH)), (2, dict(threads=64)),
    (2, dict(estimators=rt.EST_PATHLENGTH)), (4, dict(walk=rt.WALK_PATH)), (2, dict(images=True))])
def test_same_spectrum_wherever_it_is_kept(S, kw, bins, dirs):
    kw = dict(kw)
    nu = w.frequency_edges(bins)
    sp = (w.two_species(nu) + [w.grey_species(bins, 0.6, 0.4), w.grey_species(bins, 0.2, 0.9)])[:S]
    m = w.uniform_box_model(6, bins, 3.0, sp, max_level=1, refine=w.sphere_refine_fn(6, 0.5),
                            n_sed_dirs=dirs)
    n = 50_000
    with rt.Grid(m) as g:
        g.emit_star(n)
        g.set_frozen_temperatures(frozen_field(m))
        if kw.pop("images", False):
            pob = np.full(bins, -1, np.int32)
            pob[bins // 2] = 0
            g.set_images((0.0, math.sin(0.5), math.cos(0.5)), pob, 9, 9, 1.05 * m.half_size)
        seen = []
        for blocks in (0, 1, 3):
            g.reset()
            g.transport(n, seed=8, mode=rt.REEMIT_FROZEN, blocks_per_sm=blocks, **kw)
            c, sed = g.counters(), g.sed()[0]
            assert c["errors"] == 0 and c["emitted"] == n == c["escaped"] == int(sed[0].sum())
            seen.append((sed, g.counts(), c))
        for sed, counts, c in seen[1:]:
            assert np.array_equal(sed, seen[0][0]) and np.array_equal(counts, seen[0][1])
            assert c == seen[0][2]
