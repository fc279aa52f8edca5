"""Temperatures from counts set by the caller, over all table rows and many orders of count and
density, for one to five species (the compiled and the generic loop), refined cells, and cells
that are empty or never absorbed: against the oracle, which inverts the exact S(T). With 16384
rows an interval is 2.6e-3 in ln S, so the log-log interpolation is off by its square over 8
times the curvature of ln T(ln S) (below 1): 8.5e-7, with FP32 rounding within 1e-6."""
import dataclasses

import numpy as np
import pytest

import oracle
from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 2, 3, 4, 5])
def test_temperatures_over_all_rows(S):
    nu = w.frequency_edges(40)
    sp = (w.two_species(nu) + [w.grey_species(40, 0.6, 0.4), w.grey_species(40, 0.2, 0.9),
                               w.grey_species(40, 1.0)])[:S]
    m = w.uniform_box_model(5, 40, 1.0, sp, max_level=2, refine=w.sphere_refine_fn(5, 0.5))
    rng = np.random.default_rng(S)
    rho = m.rho * 10.0 ** rng.uniform(-7, 5, m.rho.shape)
    rho[:, ::7] = 0.0
    m = dataclasses.replace(m, rho=rho)
    cnt = np.floor(10.0 ** rng.uniform(0, 12, rho.shape)).astype(np.uint64)
    cnt[:, 3::11] = 0
    with rt.Grid(m, n_temp=16384) as g:
        g.emit_star(10_000)
        g.transport(16, seed=1)           # the tables are built by the first run
        _, eps = g.sed()
        g.set_counts(cnt)
        T = g.temperatures().astype(np.float64)
    To = oracle.temperatures(m, cnt, eps)
    assert np.all(T[(cnt == 0) | (rho == 0)] == 0.0)
    inside = (To > 1.001) & (To < 2999.0) & (cnt > 0) & (rho > 0)
    assert inside.sum() > 100
    np.testing.assert_allclose(T[inside], To[inside], rtol=1e-6)
    assert np.all(T[(To >= 3001.0) & (cnt > 0) & (rho > 0)] == 3000.0)
