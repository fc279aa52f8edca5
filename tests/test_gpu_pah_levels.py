"""The per-cell exact PAH emission at the sizes where its kernel's blocks end (levels in
blocks of 8, the register forms of 8, 24 and 56 blocks, level grids beyond them; bins in
groups of 4; fewer coarse bins than 64; ragged numbers of cells), against the FP64 oracle;
and the surrogate's pass over several PAHs at odd bin counts, against its formula.

Tolerance of the exact emission: populations are sums of positive terms in FP32, each level
a correctly rounded quotient of a sum whose roundings are a few 2^-24 of it; they add up
along the levels, at worst M of them, so 4 M 2^-24 (1e-4 for 400 levels) bounds the error of
a bin, and the FP32 table of level spectra adds 2^-24."""
import numpy as np
import pytest

from oracle import pah
from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu


def _model(bins, n_base=4, sizes=(30, 200)):
    nu = w.frequency_edges(bins)
    sp = w.two_species(nu) + [w.pah_species(nu, n) for n in sizes]
    fr = [0.7, 0.25] + [0.05 / len(sizes)] * len(sizes)
    return w.sphere_model(n_base=n_base, n_bins=bins, tau_v=3.0, species=sp, fractions=fr)


@pytest.mark.parametrize("levels,bins", [(16, 7), (17, 64), (64, 65), (65, 33), (192, 66),
                                         (400, 130), (448, 64), (449, 64), (700, 31)])
def test_exact_emission_sizes(levels, bins):
    m = _model(bins)
    N = 200_000
    with rt.Grid(m, pah_levels=levels) as g:
        g.emit_star(N)
        g.transport(N, seed=3)
        tal = g.pah_absorbed().astype(np.float64)
        _, eps = g.sed()
        J, _ = g.pah_emission()
        # a ragged part of the cells, and one PAH
        part, _ = g.pah_emission(first=5, n=min(43, g.N - 5))
        one, _ = g.pah_emission(pah=1)
    assert np.array_equal(part, J[5:5 + part.shape[0]])
    V = (2 * m.half_size / m.tree.n_base) ** 3
    K = min(64, bins)
    e = pah.coarse_photon_energy(m.nu_edges, K)
    tabs = [pah.level_tables(s.kabs * s.mol_mass, s.modes, m.nu_edges, n_levels=levels)
            for s in m.species[2:]]
    cells = np.nonzero(tal.sum(axis=(0, 2)) > 0)[0]
    assert len(cells) > 20
    for c in cells[:: max(1, len(cells) // 4)]:
        want = []
        for p in range(2):
            s = m.species[2 + p]
            n_mol = m.rho[2 + p, c] * V / s.mol_mass
            R = pah.cell_rates(tal[p, c], eps, n_mol, e)
            want.append(n_mol * pah.emission(pah.populations(R, e, tabs[p])[0], tabs[p])
                        if R.any() else np.zeros(bins))
        for got, ref in ((J[c], want[0] + want[1]), (one[c], want[1])):
            # bins below 1e-6 of the peak come from levels whose FP32 populations run out
            big = ref > 1e-6 * ref.max()
            np.testing.assert_allclose(got[big], ref[big], rtol=4 * levels * 2.0 ** -24 + 1e-6)


@pytest.mark.parametrize("bins,sizes", [(31, (50,)), (64, (30, 200)), (257, (30, 100, 200)),
                                        (300, (30, 60, 120, 200))])
def test_surrogate_rows(bins, sizes):
    torch = pytest.importorskip("torch")
    m = _model(bins, sizes=sizes)
    N = 100_000
    net = rt.MLP(min(64, bins) + 2, 64, 2, bins, seed=3)
    with rt.Grid(m) as g:
        g.emit_star(N)
        g.transport(N, seed=3)
        J, nf = g.pah_emission(mode=rt.PAH_SURROGATE, surrogate=net)
        auto, na = g.pah_emission(mode=rt.PAH_AUTO, surrogate=net, tol=1e9)
        exact, _ = g.pah_emission()
        none, n_all = g.pah_emission(mode=rt.PAH_AUTO, surrogate=net, tol=-1.0)
        has = g.pah_absorbed().sum(axis=(0, 2)) > 0
        want = np.zeros((g.N, bins))
        beyond = np.zeros(g.N, bool)  # an untrained network's sums can exceed any tolerance
        for p in range(g.n_pah):
            X = torch.zeros((g.N, g.n_coarse + 2), device="cuda")
            Y, pa = torch.zeros((g.N, bins), device="cuda"), torch.zeros(g.N, device="cuda")
            g.pah_training_pairs(p, X, Y, pa)
            net.forward(X, Y)
            q = torch.clamp(torch.exp(7.0 * (Y.double() - 1.0)) - 1e-6, min=0.0)
            row = pa[:, None] * q / q.sum(dim=1, keepdim=True)
            beyond |= ((pa > 0) & ((q.sum(dim=1) - 1).abs() > 1e9)).cpu().numpy()
            want += torch.where(pa[:, None] > 0, row, torch.zeros_like(row)).cpu().numpy()
    assert nf == 0 and na == int(beyond.sum()) and n_all == int(has.sum())
    # exp and the sums round in FP32: a few 2^-24 times the exponent (|7 (y - 1)| < 30)
    np.testing.assert_allclose(J, want, rtol=1e-5, atol=1e-6 * want.max())
    assert np.array_equal(auto, np.where(beyond[:, None], exact, J))
    assert np.array_equal(none, exact)
