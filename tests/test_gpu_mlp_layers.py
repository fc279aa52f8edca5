"""The layer kernels of training and of networks too wide for the fused forward, at the
edges of their tiles (128 rows, 64 columns, 256 of the contraction, 64 rows of a gradient
split) and of the padding to 16, against the same network in PyTorch FP32 with the
operands rounded to BF16 where the kernels round them.

Tolerance: the kernels' sigmoid is the hardware's (2^-11) and their sums run in another
order, so an activation or a gradient passed down may round to the neighbouring BF16 value,
a step of at most 2^-8 of it; a weight gradient is a sum of products of two of them, hence
2 x 2^-8 = 8e-3 of its norm at the very most, 1e-2 with the FP32 sums."""
import numpy as np
import pytest

from paper_1201_3588_gb300 import rt

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _bf(x):
    return x.to(torch.bfloat16).float()


def _layers(p, dims):
    out, o = [], 0
    for a, b in zip(dims[:-1], dims[1:]):
        out.append((p[o:o + a * b].view(b, a), p[o + a * b:o + a * b + b]))
        o += a * b + b
    return out


def _reference(p, dims, x, t):
    """Output, loss and gradients with BF16 operands and FP32 sums."""
    a, zs, acts = _bf(x), [], []
    ls = _layers(p, dims)
    for i, (W, b) in enumerate(ls):
        acts.append(a)
        z = a @ _bf(W).T + b
        zs.append(z)
        a = _bf(z * torch.sigmoid(z)) if i + 1 < len(ls) else z
    e = a - t
    dz, grads = 2 * e / e.numel(), []
    for i in range(len(ls) - 1, -1, -1):
        grads = [(_bf(dz).T @ acts[i]).reshape(-1), dz.sum(0)] + grads
        if i:
            s = torch.sigmoid(zs[i - 1])
            dz = (_bf(dz) @ _bf(ls[i][0])) * s * (1 + zs[i - 1] * (1 - s))
    return a, float((e ** 2).mean()), grads


@pytest.mark.parametrize("M,n_in,hidden,layers,n_out", [
    (1, 1, 16, 1, 1), (63, 17, 64, 2, 33), (64, 66, 256, 3, 200), (65, 66, 100, 2, 63),
    (127, 80, 48, 1, 65), (129, 255, 272, 2, 128), (1024, 66, 256, 3, 200),
    (1000, 300, 520, 2, 300), (20_011, 49, 128, 2, 131)])
def test_layer_kernels(M, n_in, hidden, layers, n_out):
    torch.backends.cuda.matmul.allow_tf32 = False
    dims = [n_in] + [hidden] * layers + [n_out]
    net = rt.MLP(n_in, hidden, layers, n_out, seed=1)
    rng = np.random.default_rng(M)
    p = net.get_params() + rng.uniform(-0.1, 0.1, net.n_params).astype(np.float32)
    net.set_params(p)
    x = torch.from_numpy(rng.normal(size=(M, n_in)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.normal(size=(M, n_out)).astype(np.float32)).cuda()
    y_ref, loss_ref, g_ref = _reference(torch.from_numpy(p).cuda(), dims, x, t)
    y = torch.full((M, n_out), float("nan"), device="cuda")
    net.forward(x, y)
    assert float((y - y_ref).norm()) < 1e-2 * float(y_ref.norm())
    for _ in range(2):  # the second pass finds the first one's buffers
        loss, g = net.loss_grad(x, t, want_grad=True)
        assert abs(loss / loss_ref - 1) < 1e-2
        g = torch.from_numpy(g).cuda()
        o = 0
        for i, ref in enumerate(g_ref):
            n = ref.numel()
            err = float((g[o:o + n] - ref).norm()) / max(float(ref.norm()), 1e-20)
            assert err < 1e-2, (i, err)
            o += n
    # one Adam step from zero moments moves every parameter by lr g / (|g| + eps)
    net.adam_step(1e-3)
    step = torch.from_numpy(net.get_params() - p).cuda()
    want = -1e-3 * g / (g.abs() + 1e-8)
    # the step is lost in the rounding of p (2^-24 |p|) and of the moments (a few 2^-24)
    assert float((step - want).abs().max()) < 1e-3 * 1e-4 + 2.0 ** -23 * float(np.abs(p).max())
