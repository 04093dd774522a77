"""BF16 gradient of a network whose weight-gradient tiles fill the device by themselves:
few copies of the gradient in the workspace, and the same products.  Reference and
tolerance as for the tile edges: the network in FP64 with every GEMM operand rounded to
BF16, 2e-3 of the largest entry of each layer's gradient.  Memory: the buffers a batch
needs (BF16 and FP32 activations and gradients, 16 bytes a unit) and four gradient copies.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nin,width,nout,batch", [(64, 2048, 64, 4096), (48, 700, 225, 1000)])
def test_wide_network(nin, width, nout, batch):
    from paper_2510_24968_gb300.guess import GuessNet

    g = torch.Generator(device="cuda").manual_seed(width)
    r = lambda *s: torch.randn(*s, generator=g, device="cuda")  # noqa: E731
    shapes = [(nin, width), (width,), (width, width), (width,), (width, nout), (nout,)]
    P = [r(*s) / (s[0] ** 0.5 if len(s) == 2 else 10.0) for s in shapes]
    net = GuessNet(nin=nin, width=width, nout=nout, params=torch.cat([p.reshape(-1) for p in P]).cpu().numpy())
    x, t = r(batch, nin), r(batch, nout)
    mask = (torch.rand(batch, nout, generator=g, device="cuda") < 0.5).float()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    loss, grad = net.grad(x.data_ptr(), t.data_ptr(), mask.data_ptr(), batch, bf16=True)
    used = free - torch.cuda.mem_get_info()[0]
    assert used < 16 * batch * (nin + 2 * width + nout + 192) + 4 * 4 * sum(p.numel() for p in P) + (32 << 20)
    assert np.array_equal(grad, net.grad(x.data_ptr(), t.data_ptr(), mask.data_ptr(), batch, bf16=True)[1])

    q = lambda v: v.float().to(torch.bfloat16).double()  # noqa: E731
    W1, b1, W2, b2, W3, b3 = (p.double() for p in P)
    z1 = q(x) @ q(W1) + b1
    h1 = z1 * torch.sigmoid(z1)
    z2 = q(h1) @ q(W2) + b2
    h2 = z2 * torch.sigmoid(z2)
    y = q(h2) @ q(W3) + b3
    dy = 2 * mask.double() * (y - t) / mask.double().sum()
    back = lambda d, z: d * torch.sigmoid(z) * (1 + z * (1 - torch.sigmoid(z)))  # noqa: E731
    d2 = back(q(dy) @ q(W3).T, z2)
    d1 = back(q(d2) @ q(W2).T, z1)
    want = [q(x).T @ q(d1), d1.sum(0), q(h1).T @ q(d2), d2.sum(0), q(h2).T @ q(dy), dy.sum(0)]
    assert loss == pytest.approx(float((mask * (y - t) ** 2).sum() / mask.sum()), rel=1e-3)
    at = 0
    for w in want:
        got = torch.from_numpy(grad[at:at + w.numel()].copy()).reshape(w.shape).double()
        at += w.numel()
        assert (got - w.cpu()).abs().max() <= 2e-3 * w.abs().max().cpu()
