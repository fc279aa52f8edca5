"""The surrogate's pass beside a full device: where the rows of all active cells do not fit, it
runs over smaller batches, with the same result (the rows are independent of one another)."""
import pytest

from paper_1201_3588_gb300 import rt, workloads as w
from _helpers import frozen_field

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

MB = 1 << 20


def _grid(m, n):
    g = rt.Grid(m)
    g.emit_star(n)
    g.set_frozen_temperatures(frozen_field(m))
    g.transport(n, seed=3, mode=rt.REEMIT_FROZEN)
    return g


def _fill(leave):
    """Device memory down to `leave` bytes."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog = []
    while True:
        free = torch.cuda.mem_get_info()[0]
        if free <= leave + 2 * MB:
            return hog
        try:
            hog.append(torch.empty((free - leave) // (2 * MB) * 2 * MB, dtype=torch.uint8,
                                   device="cuda"))
        except torch.OutOfMemoryError:       # in pieces: what is left is not contiguous
            leave += 8 * MB


@pytest.mark.parametrize("mode", [rt.PAH_SURROGATE, rt.PAH_AUTO])
def test_smaller_batches_beside_a_full_device(mode):
    bins, sizes = 1024, (30, 60, 120, 200)
    nu = w.frequency_edges(bins)
    sp = w.two_species(nu) + [w.pah_species(nu, n) for n in sizes]
    m = w.sphere_model(n_base=28, n_bins=bins, tau_v=3.0, species=sp,
                       fractions=[0.7, 0.25] + [0.0125] * 4)
    net = rt.MLP(64 + 2, 64, 2, bins, seed=3)
    n = 1_000_000
    kw = dict(mode=mode, surrogate=net, tol=1e9)
    with _grid(m, n) as g, _grid(m, n) as tight:
        out = [torch.zeros((g.N, bins), device="cuda") for _ in range(2)]
        _, nf = g.pah_emission(out=out[0], **kw)
        tight.pah_emission(out=out[1])       # builds what does not depend on the network
        out[1].zero_()
        active = len(tight.pah_emission_active()[0])
        need = 4 * active * (66 + bins) * 4
        assert need > 150 * MB
        hog = _fill(need // 3)
        try:
            _, nf_tight = tight.pah_emission(out=out[1], **kw)
        finally:
            del hog
            torch.cuda.empty_cache()
        assert nf_tight == nf
        assert torch.equal(out[0], out[1])
        # room again: the whole list in one batch
        out[1].zero_()
        tight.pah_emission(out=out[1], **kw)
        assert torch.equal(out[0], out[1])
