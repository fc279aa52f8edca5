"""The forward pass when a wait for the tensor cores runs out (a limit of 0 gives up every
wait of the epilogue at once, while weight copies and products are on their way): the kernel
ends by itself with its copies and products landed and its tensor memory given back, the next
read of the handle reports the timeout, and the GPU goes on computing as before."""
import pytest

from paper_1201_3588_gb300 import rt, workloads as w

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RT_ERR_TIMEOUT = 4
# rows for the kernel of many rows (more than 152 tiles of 128, output rows on 32-byte
# boundaries): one and several steps a CTA, one and several layers and output chunks
MANY = [(39_000, 66, 256, 3, 200), (150_001, 66, 256, 3, 200), (90_000, 34, 64, 1, 8),
        (60_000, 128, 128, 2, 400)]

# and for the one of few rows or ragged outputs: one and several tiles a CTA
FEW = [(100, 66, 256, 3, 200), (45_001, 66, 256, 3, 131), (60_000, 34, 64, 1, 7),
       (30_000, 128, 128, 2, 333)]


def _net(n_in, hidden, layers, n_out):
    return rt.MLP(n_in, hidden, layers, n_out, seed=3)


@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", MANY + FEW)
def test_gives_up_reports_and_goes_on(M, n_in, hidden, layers, n_out):
    x = torch.randn((M, n_in), generator=torch.Generator().manual_seed(1)).cuda()
    good, bad = _net(n_in, hidden, layers, n_out), _net(n_in, hidden, layers, n_out)
    want = good.forward(x, torch.empty((M, n_out), device="cuda")).clone()
    bad.set_wait_limit(0.0)
    y = torch.zeros((M, n_out), device="cuda")
    for _ in range(3):
        bad.forward(x, y)
    torch.cuda.synchronize()
    with pytest.raises(rt.RTError) as e:
        bad.get_params()
    assert e.value.code == RT_ERR_TIMEOUT
    # tensor memory that was not given back would leave none for these
    for net in (good, _net(n_in, hidden, layers, n_out)):
        got = net.forward(x, torch.zeros((M, n_out), device="cuda"))
        torch.cuda.synchronize()
        net.get_params()
        assert torch.equal(got, want)
    # within the limit again: the outputs are those of any other handle
    bad.set_wait_limit(2.0)
    assert torch.equal(bad.forward(x, y), want)


@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", MANY + FEW)
def test_no_row_keeps_what_it_held(M, n_in, hidden, layers, n_out):
    x = torch.randn((M, n_in), generator=torch.Generator().manual_seed(1)).cuda()
    net = _net(n_in, hidden, layers, n_out)
    net.set_wait_limit(0.0)
    # y as an earlier, plausible result, between guards
    buf = torch.full((M * n_out + 16,), 0.5, device="cuda")
    y = buf[8:8 + M * n_out].view(M, n_out)
    net.forward(x, y)
    torch.cuda.synchronize()
    assert torch.isnan(y).all()
    assert (buf[:8] == 0.5).all() and (buf[8 + M * n_out:] == 0.5).all()


@pytest.mark.parametrize("mode", [rt.PAH_SURROGATE, rt.PAH_AUTO])
@pytest.mark.parametrize("n_base", [4, 36])        # few rows, and enough for the other kernel
def test_emission_reports_it(mode, n_base):
    nu = w.frequency_edges(64)
    sp = w.two_species(nu) + [w.pah_species(nu, n) for n in (30, 200)]
    m = w.sphere_model(n_base=n_base, n_bins=64, tau_v=3.0, species=sp,
                       fractions=[0.7, 0.25, 0.025, 0.025])
    net = rt.MLP(64 + 2, 64, 2, 64, seed=3)
    n = 1_000_000 if n_base > 4 else 100_000
    with rt.Grid(m) as g:
        g.emit_star(n)
        g.transport(n, seed=3)
        rows = 2 * len(g.pah_emission_active(mode=rt.PAH_EXACT)[0])
        assert (rows > 152 * 128) == (n_base > 4)
        want, _ = g.pah_emission(mode=mode, surrogate=net, tol=1e9)
        again, _ = g.pah_emission(mode=mode, surrogate=net, tol=1e9)
        assert (want == again).all()
        net.set_wait_limit(0.0)
        for call in (g.pah_emission, g.pah_emission_active):
            with pytest.raises(rt.RTError) as e:
                call(mode=mode, surrogate=net, tol=1e9)
            assert e.value.code == RT_ERR_TIMEOUT
        # another handle, and the exact solution, are not affected
        fresh, _ = g.pah_emission(mode=mode, surrogate=rt.MLP(64 + 2, 64, 2, 64, seed=3), tol=1e9)
        assert (fresh == want).all()
        g.pah_emission()


def test_limit_is_checked():
    net = _net(8, 16, 1, 8)
    for s in (-1.0, float("nan"), 61.0):
        with pytest.raises(rt.RTError):
            net.set_wait_limit(s)
