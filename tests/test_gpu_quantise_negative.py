"""FP64 positions in a box centred on zero: the deposit stays bit-exact against
the oracle's division, and takes no longer than for positions in [0, L)."""
import numpy as np
import pytest

from oracle import pm_oracle as O
from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,box", [(16, 16.0), (64, 333.333), (192, 7.0e-3), (128, 1.0e6)])
def test_negative_edges_of_cells_and_weights(n, box):
    import torch
    rng = np.random.default_rng(n + 1)
    d = box / n
    x = -rng.integers(0, 3 * n * 65536, 5000) * (d / 65536.0)
    x = np.concatenate([x, np.nextafter(x, np.inf), np.nextafter(x, -np.inf), -np.arange(n) * d, rng.uniform(-box / 2, box / 2, 9001),
                        -box * 10.0 ** rng.uniform(-12, 2, 2000), [-d * 3.2e4, -d * 3.3e4, -1e-300, -5e-324]])
    pos = np.stack([rng.permutation(x) for _ in range(3)])
    pm = nupm.PM(n, pos.shape[1], box, 0.3, 0.0, n_kbins=8, precision="fp64", flags=nupm.PM_KEEP_DEPOSIT)
    pm.deposit(torch.from_numpy(pos).cuda())
    F = pm.field(nupm.FIELD_DEPOSIT).cpu().numpy()
    pm.check()
    pm.close()
    c, w = O.quantise_positions_f64(pos, box, n)
    assert np.array_equal(F.view(np.uint64).astype(np.int64), O.cic_deposit(c, w, n))


def test_a_centred_box_takes_no_longer():
    import torch
    n, ms = 256, []
    pm = nupm.PM(n, n ** 3, 500.0, 0.3, 0.0, n_kbins=8, precision="fp64")
    x = torch.rand((3, n ** 3), dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(1)) * 500.0
    for pos in (x, (x - 250.0).contiguous()):
        best = float("inf")
        for _ in range(5):
            pm.timing(True)
            pm.deposit(pos)
            best = min(best, pm.get_timing()["deposit"][0])
        ms.append(best)
    pm.check()
    pm.close()
    assert ms[1] < 1.3 * ms[0], ms        # the division for every negative coordinate: over twice as long
