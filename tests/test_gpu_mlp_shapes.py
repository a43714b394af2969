"""The prefilter network at the edges of its tiles (64 rows a tile, two tiles a CTA, 64 rows
a stage of the weight gradients): logits do not depend on the batch or the alignment they are
computed in, and gradients match a float64 reference on the same bf16 operands.

Tolerance of the gradients: 2e-3 of the largest entry, as for the small batch of
test_gpu_prefilter.py.  The reference takes the kernel's own logits (compared with a
reference there) and forms dz in float32, so that the roundings of dh2 to bf16, each 2^-8
of a term, fall the same way on both sides; with few rows one such term is the entry."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import paper_2009_14467_gb300 as P
    from paper_2009_14467_gb300 import prefilter as F
    ctx = P.Context(0)
    yield F, ctx
    ctx.close()


def _x(n, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randn((n, 16), generator=g).bfloat16().cuda()


def test_logits_do_not_depend_on_the_batch(env):
    F, ctx = env
    net = F.MLP(seed=3)
    x = _x(152 * 128 * 2 + 77, 1)
    z = F.forward(ctx, net, x)
    for n in (1, 2, 31, 127, 128, 129, 255, 257, 4097, 152 * 128, 152 * 128 + 1):
        assert torch.equal(F.forward(ctx, net, x[:n].contiguous()), z[:n]), n
    odd = torch.empty(1 + 1000 * 16, dtype=torch.bfloat16, device="cuda")
    odd[1:] = x[:1000].reshape(-1)
    assert torch.equal(F.forward(ctx, net, odd[1:].view(1000, 16)), z[:1000])


@pytest.mark.parametrize("n", [1, 31, 33, 127, 129, 2433, 20000])
def test_gradients_at_tile_edges(env, n):
    F, ctx = env
    net = F.MLP(seed=4)
    x = _x(n, n)
    y = (torch.rand(n, generator=torch.Generator().manual_seed(n)) < 0.3).float().cuda()
    loss = torch.zeros(1, device="cuda")
    zf = F.forward(ctx, net, x)
    F.train_step(ctx, net, x, y, 0.0, 3.0, loss)
    xd, yd = x.double(), y.double()
    w1, w2, w3 = net.w1b.double(), net.w2b.double(), net.w3b.double()

    def r(t):
        return t.float().bfloat16().double()

    h1 = r(torch.relu(xd @ w1 + net.b1.double()))
    h2 = r(torch.relu(h1 @ w2 + net.b2.double()))
    z = zf.double()
    w = torch.where(yd > 0.5, 3.0, 1.0)
    dz = (w.float() * (torch.sigmoid(zf) - y) / n).double()
    d2 = r(torch.where(h2 > 0, dz[:, None] * w3, 0.0))
    d1 = torch.where(h1 > 0, d2 @ w2.T, 0.0)
    want = [xd.T @ r(d1), d1.sum(0), h1.T @ d2, d2.sum(0), h2.T @ dz, dz.sum().reshape(1)]
    for got, ref in zip(net.grads(), want):
        scale = max(float(ref.abs().max()), 1e-12)
        assert float((got.double() - ref).abs().max()) <= 2e-3 * scale
    ref = (w * (torch.nn.functional.softplus(z) - yd * z)).mean()
    assert abs(float(loss) - float(ref)) <= 2e-3 * abs(float(ref))
