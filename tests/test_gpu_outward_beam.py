"""A beam that starts on the boundary and points out of the domain: every package leaves as it
is drawn, so a warp that has just drawn 32 has none to walk. All packages are emitted and
escape into the direct spectrum, with and without the path-length tally, for more packages
than there are lanes."""
import pytest

from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("estimators", [0, rt.EST_PATHLENGTH])
@pytest.mark.parametrize("S", [1, 2, 4])
def test_every_package_is_drawn(S, estimators):
    nu = w.frequency_edges(16)
    sp = (w.two_species(nu) + [w.grey_species(16, 0.6, 0.4), w.grey_species(16, 0.2, 0.9)])[:S]
    m = w.uniform_box_model(4, 16, 2.0, sp)
    beam = w.Star(pos_cm=(0.0, 0.0, m.half_size), beam_dir=(0.1, 0.2, 0.97), kind=w.SOURCE_BEAM)
    n_all = 400_000
    with rt.Grid(m) as g:
        g.emit_star(n_all, star=beam)
        for n, kw in ((n_all, {}), (1, {}), (33, {}), (5_000, dict(threads=32, blocks_per_sm=1)),
                      (n_all, dict(refill_period=1))):
            g.reset()
            g.transport(n, seed=3, estimators=estimators, **kw)
            c, sed = g.counters(), g.sed()[0]
            assert c["emitted"] == n == c["escaped"], (n, kw, c)
            assert int(sed[0].sum()) == n == int(sed[1].sum())
            assert c["errors"] == 0 == c["absorptions"] + c["scatters"] + c["crossings"]
            assert not g.counts().any()
            if estimators:
                assert not g.pathlength().any()
