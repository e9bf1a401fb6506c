"""Forces by sorted slot where a few grid rows hold much of the mass: the tiles'
parts beyond the first, bit for bit, on either side of the particle numbers between
which tiles are taken; and no waiting for the few CTAs that own those rows."""
import numpy as np
import pytest

from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


def _box(n, npart, share, seed):
    """`share` of the particles in one filament along x, sigma one cell, the rest even."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((3, npart), generator=g, device="cuda", dtype=torch.float64) * n
    k = int(share * npart)
    x[1:, :k] = (n / 2 + torch.randn((2, k), generator=g, device="cuda", dtype=torch.float64)) % n
    cell = torch.floor(x)
    off = (x - cell).float().clamp_(max=1 - 2.0 ** -24)
    return torch.cat([cell.to(torch.int32), off.view(torch.int32)]).contiguous()


def _forces(pm, pos, rows):
    import torch
    pm.set_tuning(gather_rows=rows)
    vel = torch.zeros((3, pos.shape[1]), device="cuda")
    acc = torch.full_like(vel, float("nan"))
    pm.deposit(pos)
    pm.nu_response(0.1, None, None)
    pm.kick(pos, vel, 0.1, 0.5, acc_out=acc)
    return acc, vel


@pytest.mark.parametrize("n,npart,share", [(128, 128 ** 3 // 2 - 1, 0.5), (128, 128 ** 3 // 2, 0.5), (128, 2 ** 21 + 77, 0.9),
                                           (192, 192 ** 3 // 2 + 5, 0.5), (256, 2 ** 23, 0.5), (256, 2 ** 24 + 1, 0.02),
                                           (512, 2 ** 26 + 3, 0.3), (1024, 2 ** 20, 0.5),
                                           (16, 32768, 0.5), (16, 32769, 0.5), (32, 65536, 0.9), (64, 65536, 0.5),
                                           (64, 65537, 0.5), (192, 20011, 0.9), (256, 65536, 0.5), (256, 1, 0.0),
                                           (512, 32768, 0.5), (512, 32769, 0.5)])
def test_parts_are_bit_identical(n, npart, share):
    import torch
    pm = nupm.PM(n, npart, 100.0, 0.3, 0.0, n_kbins=8, precision="fp32")
    pos = _box(n, npart, share, n)
    ref, got = _forces(pm, pos, 0), _forces(pm, pos, 2)
    assert torch.equal(got[0], ref[0]) and torch.equal(got[1], ref[1])
    pm.check()
    pm.close()


@pytest.mark.parametrize("n", [128, 256])
def test_a_filament_takes_no_longer_than_an_even_box(n):
    import torch
    npart = n ** 3
    pm = nupm.PM(n, npart, 100.0, 0.3, 0.0, n_kbins=8, precision="fp32")
    ms = []
    for share in (0.0, 0.5):
        pos = _box(n, npart, share, n)
        vel = _forces(pm, pos, 2)[1]
        best = float("inf")
        for _ in range(5):
            pm.timing(True)
            pm.kick(pos, vel, 0.1, 0.5)
            best = min(best, pm.get_timing()["interp"][0])
        ms.append(best)
    pm.check()
    pm.close()
    assert ms[1] < 2.0 * ms[0], ms   # one CTA for all of a tile: 10 times as long
