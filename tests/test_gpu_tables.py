"""The FP64 tables at the sizes where their kernels' tiles end (31 and 32 bins per warp
pass, one bin, the most bins; few temperature rows), against the oracle: temperatures
inverted from the same counts, frozen-mode histories, and the temperature distribution
of a PAH heated by single photons."""
import numpy as np
import pytest

import oracle
from oracle import pah
from paper_1201_3588_gb300 import rt, workloads as w
from _divergence import explain
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
EV = 1.602176634e-12


@pytest.mark.parametrize("bins", [1, 2, 31, 32, 33, 63, 1024])
def test_tables_against_oracle(bins):
    m = w.sphere_model(n_base=4, n_bins=bins, tau_v=2.0)
    N, Tf = 20_000, frozen_field(m)
    ids = np.arange(60, dtype=np.uint64) * 7
    with rt.Grid(m) as g:
        g.emit_star(N)
        g.set_frozen_temperatures(Tf)
        cats, bad = explain(g, m, ids, Tf, 5, N)
        g.transport(N, seed=5)
        cnt, T, (_, eps) = g.counts(), g.temperatures(), g.sed()
    To = oracle.temperatures(m, cnt, eps)
    pos = (To > 1.0) & (To < 2900.0)
    # the table's log-log interpolation between rows 0.8 % apart in T
    np.testing.assert_allclose(T[pos], To[pos], rtol=2e-4)
    # histories: bins come from the tables on the GPU and from exact spectra in the
    # oracle, so a history may part where the table's resolution says so, and only there
    assert not bad, (cats, bad)


def test_few_temperature_rows():
    m = w.sphere_model(n_base=4, n_bins=33, tau_v=2.0)
    with rt.Grid(m, n_temp=3, t_min=5.0, t_max=500.0) as g:
        g.emit_star(5000)
        g.transport(5000, seed=5)
        T, c = g.temperatures(), g.counters()
    assert c["errors"] == 0 and c["escaped"] == 5000
    assert np.isfinite(T).all() and T.max() <= 500.0


@pytest.mark.parametrize("bins,levels", [(1, 16), (30, 17), (31, 33), (32, 64), (62, 100),
                                         (63, 31), (1024, 40)])
def test_distribution_sizes(bins, levels):
    nu = w.frequency_edges(bins)
    sp = w.pah_species(nu, 50)
    sig = sp.kabs * sp.mol_mass
    cases = [dict(modes=sp.modes, h_nu=e * EV, rate=1e-3, t_top=3000.0)
             for e in (3.8, 40.0, 1000.0)]
    P, T, a, em = rt.pah_temperature_distribution(cases, nu, np.array([sig] * 3),
                                                  n_levels=levels, t_sub=1500.0)
    for i, c in enumerate(cases):
        r = pah.temperature_distribution(sp.modes, sig, nu, c["h_nu"], c["rate"] * c["h_nu"],
                                         1.0, n_levels=levels, t_top=3000.0, t_sub=1500.0)
        np.testing.assert_allclose(T[i], r["T"], rtol=1e-11)
        big = r["P"] > 1e-6 * r["P"].max()
        np.testing.assert_allclose(P[i][big], r["P"][big], rtol=1e-7)
        np.testing.assert_allclose(em[i], r["emission"], rtol=1e-7, atol=1e-12 * em[i].max())
        assert a[i] == pytest.approx(r["p_above"], rel=1e-7, abs=1e-15)
