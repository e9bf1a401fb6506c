"""The surrogate network at the edges of its tiles: row counts around 16 and 32,
more rows than one wave of CTAs, every input width that the padding touches.
Forward against FP64 with the same BF16 weights; gradient against autograd."""
import numpy as np
import pytest

from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_in,n", [(1, 1), (4, 15), (5, 16), (12, 17), (12, 31), (13, 33), (16, 4864), (12, 4865),
                                    (12, 30011)])
def test_forward_and_gradient(n_in, n):
    import torch
    rng = np.random.default_rng(n_in * 100003 + n)
    W = nupm.MLP_WIDTH
    cut = np.cumsum([0, W * n_in, W, W * W, W, W, 1])
    th = np.concatenate([rng.normal(size=W * n_in) / np.sqrt(n_in), 0.2 * rng.normal(size=W),
                         rng.normal(size=W * W) / 11.0, 0.2 * rng.normal(size=W), rng.normal(size=W) / 11.0,
                         [0.3]]).astype(np.float32)
    mu, sig = rng.normal(size=n_in).astype(np.float32), (0.5 + rng.random(n_in)).astype(np.float32)
    X = (rng.normal(size=(n, n_in)) * 1.5).astype(np.float32)
    y = rng.normal(size=n).astype(np.float32)
    mlp = nupm.MLP(n_in=n_in)
    mlp.set_params(th)
    mlp.set_norm(mu, sig, -0.5, 1.5)
    Xd, yd = torch.from_numpy(X).cuda(), torch.from_numpy(y).cuda()
    out = mlp.forward(Xd).cpu().numpy()
    g, loss = mlp.grad(Xd, yd)
    p = [torch.from_numpy(th[cut[i]:cut[i + 1]]) for i in range(6)]
    p = [(q.bfloat16() if i in (0, 2, 4) else q).double().requires_grad_(True) for i, q in enumerate(p)]
    xh = (torch.from_numpy(X).double() - torch.from_numpy(mu).double()) / torch.from_numpy(sig).double()
    h1 = torch.tanh(xh @ p[0].reshape(W, n_in).T + p[1])
    o = torch.tanh(h1 @ p[2].reshape(W, W).T + p[3]) @ p[4] + p[5]
    ref = torch.autograd.grad((o - (torch.from_numpy(y).double() + 0.5) / 1.5).square().mean(), p)
    gref = torch.cat(ref).numpy()
    # sums of 16, 128 and 128 FP32 terms of order one: 2^-24 x 272 bounds each output
    assert np.max(np.abs(out - (-0.5 + 1.5 * o.detach().numpy()))) < 1.5 * 272 * 2.0 ** -24
    g = g.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - gref) < 2e-6 * np.linalg.norm(gref)
    lref = float((o - (torch.from_numpy(y).double() + 0.5) / 1.5).square().mean().detach())
    assert abs(float(loss) - lref) < 2e-6 * lref
    mlp.close()
