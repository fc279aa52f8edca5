"""PAH emission on frequency grids that end in the optical, where the lowest of many levels
cool at rates that FP32 holds as denormal numbers, whose reciprocal overflows: the emission is
finite in every cell, also where one PAH absorbed nothing beside another that did, and the
emission of all PAHs is the sum of each one's (one FP32 addition: 2^-23)."""
import dataclasses

import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lam_max,levels", [(1.0, 2048), (0.8, 2048), (0.8, 400), (0.5, 700)])
@pytest.mark.parametrize("sizes", [(30, 200), (200, 100, 30)])
def test_cold_levels(lam_max, levels, sizes):
    bins = 64
    nu = w.frequency_edges(bins, 0.1, lam_max)
    sp = w.two_species(nu) + [w.pah_species(nu, n) for n in sizes]
    m = w.sphere_model(n_base=12, n_bins=bins, tau_v=1.0, species=sp,
                       fractions=[0.7, 0.25] + [0.05 / len(sizes)] * len(sizes))
    m = dataclasses.replace(m, nu_edges=nu)
    with rt.Grid(m, pah_levels=levels) as g:
        g.emit_star(20_000)
        g.transport(20_000, seed=3)
        has = g.pah_absorbed().sum(axis=2) > 0
        assert (has.any(axis=0) & ~has.all(axis=0)).sum() > 20    # some without one of them
        J, _ = g.pah_emission()
        one = [g.pah_emission(pah=p)[0] for p in range(len(sizes))]
        cells, rows, _ = g.pah_emission_active()
    assert np.isfinite(J).all() and all(np.isfinite(x).all() for x in one)
    assert (J >= 0).all() and not J[~has.any(axis=0)].any()
    for p, x in enumerate(one):
        assert not x[~has[p]].any()
    np.testing.assert_allclose(J, sum(x.astype(np.float64) for x in one),
                               rtol=len(sizes) * 2.0 ** -23)
    assert np.array_equal(rows, J[cells])
