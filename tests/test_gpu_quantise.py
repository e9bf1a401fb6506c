"""FP64 positions at the edges of the integer quantisation: the deposit stays
bit-exact against the oracle's division (exact equality of integers)."""
import numpy as np
import pytest

from oracle import pm_oracle as O
from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,box", [(16, 16.0), (32, 100.0), (64, 333.333), (192, 7.0e-3), (128, 1.0e6)])
def test_edges_of_cells_and_weights(n, box):
    import torch
    rng = np.random.default_rng(n)
    d = box / n
    k = rng.integers(0, n * 65536, 4000)
    x = k * (d / 65536.0)                                  # weight boundaries, then their neighbours
    x = np.concatenate([x, np.nextafter(x, np.inf), np.nextafter(x, -np.inf), np.arange(n) * d,
                        np.nextafter(np.arange(1, n) * d, 0), [0.0, -0.0, -1e-300, -1e-18 * box, 5e-324, 1e-300, np.nextafter(box, 0), box],
                        rng.uniform(-3 * box, 40 * box, 4000), rng.uniform(0, box, 8000),
                        box * 10.0 ** rng.uniform(-12, 9, 2000), [d * 3.0e4, d * 3.3e4, d * 2.0 ** 40]])
    pos = np.stack([rng.permutation(x) for _ in range(3)])
    pm = nupm.PM(n, pos.shape[1], box, 0.3, 0.0, n_kbins=8, precision="fp64", flags=nupm.PM_KEEP_DEPOSIT)
    pm.deposit(torch.from_numpy(pos).cuda())
    F = pm.field(nupm.FIELD_DEPOSIT).cpu().numpy()
    pm.check()
    pm.close()
    c, w = O.quantise_positions_f64(pos, box, n)
    assert np.array_equal(F.view(np.uint64).astype(np.int64), O.cic_deposit(c, w, n))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, 1e30])
def test_invalid_positions_are_reported(bad):
    import torch
    pos = np.full((3, 40), 3.25)
    pos[1, 17] = bad
    pm = nupm.PM(16, 40, 16.0, 0.3, 0.0, n_kbins=8, precision="fp64")
    pm.deposit(torch.from_numpy(pos).cuda())
    with pytest.raises(nupm.PMError):
        pm.check()
    pm.close()
