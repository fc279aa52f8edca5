"""The fused forward of many rows with its input off the 8- and 16-byte boundaries and its
output on a 32-byte one (the kernel then reads single floats, or pairs): the outputs are those
of an aligned input, bit for bit, for even and odd input widths."""
import pytest

from paper_1201_3588_gb300 import rt

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", [
    (39_001, 66, 256, 3, 200), (20_000, 34, 64, 1, 8), (45_003, 17, 128, 2, 264),
    (19_457, 256, 144, 1, 16)])
@pytest.mark.parametrize("shift", [1, 2, 3])
def test_input_off_its_boundary(M, n_in, hidden, layers, n_out, shift):
    net = rt.MLP(n_in, hidden, layers, n_out, seed=3)
    x = torch.randn(M * n_in, generator=torch.Generator().manual_seed(M)).cuda()
    want = torch.empty((M, n_out), device="cuda")
    net.forward(x.view(M, n_in), want)
    xb = torch.full((M * n_in + 8,), float("nan"), device="cuda")   # nothing beside the rows is read
    xb[shift:shift + M * n_in] = x
    y = torch.empty((M, n_out), device="cuda")
    assert y.data_ptr() % 32 == 0
    net.forward(xb[shift:shift + M * n_in].view(M, n_in), y)
    torch.cuda.synchronize()
    net.get_params()                       # reports a wait that ran out
    assert torch.equal(y, want)
