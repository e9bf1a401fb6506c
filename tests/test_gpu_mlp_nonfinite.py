"""Forward pass with weights that are not finite (a master weight past the BF16
range rounds to infinity): a unit with an infinite weight saturates and the
output stays finite, as the FP32 sum gives it; a NaN reaches the outputs."""
import numpy as np
import pytest

from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


def _net(n_in, seed):
    rng = np.random.default_rng(seed)
    W = nupm.MLP_WIDTH
    th = [rng.normal(size=W * n_in) / np.sqrt(n_in), 0.2 * rng.normal(size=W), rng.normal(size=W * W) / 11.0,
          0.2 * rng.normal(size=W), rng.normal(size=W) / 11.0, np.array([0.3])]
    return rng, [t.astype(np.float32) for t in th]


def _forward(n_in, th, X):
    import torch
    mlp = nupm.MLP(n_in=n_in)
    mlp.set_params(np.concatenate(th))
    out = mlp.forward(torch.from_numpy(X).cuda()).cpu().numpy()
    mlp.close()
    W = nupm.MLP_WIDTH
    p = [(torch.from_numpy(q).bfloat16() if i in (0, 2, 4) else torch.from_numpy(q)).double() for i, q in enumerate(th)]
    h1 = torch.tanh(torch.from_numpy(X).double() @ p[0].reshape(W, n_in).T + p[1])
    return out, (torch.tanh(h1 @ p[2].reshape(W, W).T + p[3]) @ p[4] + p[5]).numpy()


@pytest.mark.parametrize("n", [1, 16, 33, 5000])
@pytest.mark.parametrize("where", [[(0, 0)], [(127, 127)], [(5, 17), (5, 40), (77, 3), (78, 126), (79, 64)]])
def test_infinite_weights_saturate_their_unit(n, where):
    n_in = 12
    rng, th = _net(n_in, n)
    for i, (j, k) in enumerate(where):
        # past the BF16 range, or infinite; one sign a unit, and h1 of that column far from zero
        th[2][j * 128 + k] = (3.4e38 if i % 2 == 0 else np.inf) * (-1 if j % 2 else 1)
        th[1][k] = 4.0 if i % 2 == 0 else -4.0
        if j == 5:
            th[1][k] = 4.0
    X = (0.3 * rng.normal(size=(n, n_in))).astype(np.float32)
    out, ref = _forward(n_in, th, X)
    assert np.all(np.isfinite(ref))
    assert np.max(np.abs(out - ref)) < 272 * 2.0 ** -24     # sums of 16, 128 and 128 FP32 terms of order one


def test_a_nan_weight_is_seen():
    rng, th = _net(12, 7)
    th[2][9 * 128 + 9] = np.nan
    out, ref = _forward(12, th, rng.normal(size=(40, 12)).astype(np.float32))
    assert np.all(np.isnan(out)) and np.all(np.isnan(ref))


def test_opposite_infinities_of_a_unit_are_nan():
    rng, th = _net(12, 8)
    th[2][9 * 128 + 9], th[2][9 * 128 + 100] = np.inf, -np.inf
    th[1][9] = th[1][100] = 4.0
    out, _ = _forward(12, th, (0.3 * rng.normal(size=(40, 12))).astype(np.float32))
    assert np.all(np.isnan(out))
