"""Temperatures on grids on both sides of the size from which a thread takes all species of a
cell (2^18 cells), for every species count with a form of its own: a pattern of counts and
densities repeated over the grid gives the temperatures of a small grid with cells of the same
size (the same arithmetic; the cell size rounds, 2^-52 of it, before one FP32 rounding of T:
2^-22 with the last place). The number of clamped entries goes with them."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S", [1, 2, 3, 4, 8])
@pytest.mark.parametrize("n_base", [1, 7, 63, 64, 65])
def test_pattern_at_every_size(S, n_base):
    nu = w.frequency_edges(40)
    sp = (w.two_species(nu) + [w.grey_species(40, 0.1 * k, 0.5) for k in range(2, 8)])[:S]
    rng = np.random.default_rng(S)
    rho0 = 10.0 ** rng.uniform(-24, -14, (S, 125))
    rho0[:, ::7] = 0.0
    cnt0 = np.floor(10.0 ** rng.uniform(0, 10, (S, 125))).astype(np.uint64)
    cnt0[:, 3::11] = 0

    def temperatures(n):
        tree = w.build_tree(n, 0)
        i = np.arange(n ** 3) % 125
        m = w.explicit_model(tree, rho0[:, i], 40, sp, half_size_cm=n * 0.1 * w.AU)
        with rt.Grid(m) as g:
            g.emit_star(10_000)
            g.set_counts(np.ascontiguousarray(cnt0[:, i]))
            T = g.temperatures()
            return T, g.counters()["clamped"], i

    small, _, _ = temperatures(5)
    T, clamped, i = temperatures(n_base)
    np.testing.assert_allclose(T, small[:, i], rtol=2.0 ** -22)
    assert clamped == int((T == 3000.0).sum())
    assert (small > 0).any() and (small == 3000.0).any() and (small == 0).any()
