"""The guess network's BF16 gradient (tensor-core layers, split weight gradients)
at the edges of its tiles: batches around 128-row tiles and around the largest
split count, widths and outputs that are not multiples of the 64-element chunk.

Reference: the same network in FP64 with the operands of every GEMM rounded to
BF16 as the library rounds them.  FP32 accumulation moves a pre-rounding value
by ~1e-6 of its size, which flips a BF16 rounding (2^-8 relative) in ~1e-3 of
the cases at most, so the products agree to well below 2e-3 of the largest
gradient entry of their layer.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nin,width,nout,batch", [(48, 256, 225, 1), (48, 256, 225, 127), (48, 256, 225, 129),
                                                  (48, 256, 225, 4097), (48, 32, 225, 4224), (7, 130, 65, 257),
                                                  (65, 300, 3, 64), (130, 64, 128, 128)])
def test_bf16_gradient_at_tile_edges(nin, width, nout, batch):
    import torch

    from paper_2510_24968_gb300.guess import GuessNet

    g = torch.Generator().manual_seed(batch + width)
    r = lambda *s: torch.randn(*s, generator=g)  # noqa: E731
    shapes = [(nin, width), (width,), (width, width), (width,), (width, nout), (nout,)]
    P = [r(*s) / (s[0] ** 0.5 if len(s) == 2 else 10.0) for s in shapes]
    net = GuessNet(nin=nin, width=width, nout=nout, params=torch.cat([p.reshape(-1) for p in P]).numpy())
    x, t = r(batch, nin), r(batch, nout)
    mask = (torch.rand(batch, nout, generator=g) < 0.5).float()
    mask[0, 0] = 1.0
    dev = [v.cuda().contiguous() for v in (x, t, mask)]
    loss, grad = net.grad(*[v.data_ptr() for v in dev], batch, bf16=True)
    again = net.grad(*[v.data_ptr() for v in dev], batch, bf16=True)[1]
    assert np.array_equal(grad, again)

    q = lambda v: v.float().to(torch.bfloat16).double()  # noqa: E731
    W1, b1, W2, b2, W3, b3 = (p.double() for p in P)
    z1 = q(x) @ q(W1) + b1
    z2 = q(z1 * torch.sigmoid(z1)) @ q(W2) + b2
    h1, h2 = z1 * torch.sigmoid(z1), z2 * torch.sigmoid(z2)
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
        assert (got - w).abs().max() <= 2e-3 * w.abs().max()
