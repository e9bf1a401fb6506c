"""The gather orders, the tiled forces-by-slot form among them: forces
bit-identical to the storage-order gather at every grid size it takes, with
particles at the faces of the box and a crowded cell."""
import numpy as np
import pytest

from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


def _setup(n, npart, seed):
    import torch
    rng = np.random.default_rng(seed)
    pm = nupm.PM(n, npart, 100.0, 0.3, 0.0, n_kbins=8, precision="fp32")
    cell = rng.integers(0, n, (3, npart))
    k = max(1, npart // 20)
    cell[:, :k] = rng.choice([0, 1, 2, n - 3, n - 2, n - 1], (3, k))         # the periodic faces
    m = min(k, 20000)                             # one crowded cell (a node holds 65535 full weights), unwrapped
    cell[:, k:k + m] = cell[:, k:k + 1] + rng.integers(-n, 2 * n, (3, 1))
    off = np.minimum(rng.random((3, npart)).astype(np.float32), np.float32(1 - 2.0 ** -24))   # < 1 once rounded
    pos = np.concatenate([cell, off.view(np.int32)]).astype(np.int32)
    return pm, torch.from_numpy(pos).cuda()


def _kick(pm, pos, tuning=None):
    import torch
    if tuning is not None:
        pm.set_tuning(gather_rows=tuning)
    vel = torch.zeros((3, pos.shape[1]), device="cuda")
    acc = torch.full_like(vel, float("nan"))
    pm.deposit(pos)
    pm.nu_response(0.1, None, None)
    pm.kick(pos, vel, 0.1, 0.5, acc_out=acc)
    return acc, vel


@pytest.mark.parametrize("n,npart", [(16, 1500), (32, 9001), (64, 65536 * 2), (64, 262145), (128, 530000),
                                     (192, 1800001), (256, 4194305), (512, 1 << 25)])
def test_orders_are_bit_identical(n, npart):
    import torch
    pm, pos = _setup(n, npart, n)
    built_in = _kick(pm, pos)
    ref = _kick(pm, pos, tuning=0)
    for got in (built_in, _kick(pm, pos, tuning=1), _kick(pm, pos, tuning=2)):
        assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    pm.check()
    pm.close()
