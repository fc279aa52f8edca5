"""The fused forward at its edges: one or two tiles of 128 rows a step (152 SMs: more than
19456 rows), halves of 128 columns present or not, odd input widths and buffers off their
8- and 32-byte boundaries (the scalar loads and stores), against PyTorch FP32 with the
operands rounded to BF16 where the kernel rounds them.

Tolerance: the kernel's sigmoid is the hardware's (2^-11) and its sums run in another order,
so an activation may round to the neighbouring BF16 value, 2^-8 of it; an output sums many of
those with either sign. A single one is allowed 5 % of the outputs' RMS, which a misplaced
row, column or bias (an error of the RMS itself) exceeds by far, and all together 2 x 2^-8 of
their norm with 1e-2."""
import pytest

from paper_1201_3588_gb300 import rt

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _bf(x):
    return x.to(torch.bfloat16).float()


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", [
    (129, 1, 16, 1, 1), (19_456, 17, 64, 2, 33), (19_457, 17, 64, 2, 33),
    (19_585, 130, 144, 1, 136), (39_000, 255, 256, 1, 256), (38_913, 128, 128, 2, 128),
    (40_001, 66, 256, 2, 272)])
def test_fused_forward_edges(M, n_in, hidden, layers, n_out, shift):
    torch.backends.cuda.matmul.allow_tf32 = False
    net = rt.MLP(n_in, hidden, layers, n_out, seed=3)
    g = torch.Generator().manual_seed(M)
    p = torch.from_numpy(net.get_params())
    p += 0.2 * torch.rand(p.numel(), generator=g) - 0.1
    net.set_params(p.numpy())
    # contiguous, at `shift` floats past an aligned address; guard values on either side of y
    xb = torch.randn(M * n_in + 8, generator=g).cuda()
    b = 8 + shift
    yb = torch.full((M * n_out + 24,), 7.0, device="cuda")
    x = xb[shift:shift + M * n_in].view(M, n_in)
    y = yb[b:b + M * n_out].view(M, n_out)
    net.forward(x, y)
    torch.cuda.synchronize()
    net.get_params()                       # reports a wait that ran out
    a, o, dims = _bf(x), 0, [n_in] + [hidden] * layers + [n_out]
    pd = p.cuda()
    for i, (k, n) in enumerate(zip(dims[:-1], dims[1:])):
        z = a @ _bf(pd[o:o + k * n].view(n, k)).T + pd[o + k * n:o + k * n + n]
        o += k * n + n
        a = _bf(z * torch.sigmoid(z)) if i < layers else z
    assert (yb[:b] == 7.0).all() and (yb[b + M * n_out:] == 7.0).all()
    e = y - a
    assert float(e.norm()) < 1e-2 * float(a.norm())
    assert float(e.abs().max()) < 0.05 * float(a.pow(2).mean().sqrt())
