"""The deposit of node rows with so many records that a CTA's warps share them
(grids of 512 points on): the same 64-bit sums as the unfused deposit's global
adds, a wrapped sum reported, and no serial tail of one warp."""
import numpy as np
import pytest

from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


def _line(n, npart, k, precision, seed):
    """k particles in the row (y, z) = (n / 2, n - 1), the rest even."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((3, npart), generator=g, device="cuda", dtype=torch.float64) * n
    x[1, :k] = n // 2 + torch.rand(k, generator=g, device="cuda", dtype=torch.float64)
    x[2, :k] = n - 1 + torch.rand(k, generator=g, device="cuda", dtype=torch.float64)
    if precision == "fp64":
        return x.contiguous()                       # box = n: unit cells
    cell = torch.floor(x)
    off = (x - cell).float().clamp_(max=1 - 2.0 ** -24)
    return torch.cat([cell.to(torch.int32), off.view(torch.int32)]).contiguous()


# just below and above the records of a shared row (32768) and of one that can wrap (65536), and far above
@pytest.mark.parametrize("precision,n", [("fp32", 512), ("fp64", 512), ("fp32", 1024), ("fp32", 256)])
@pytest.mark.parametrize("k", [32000, 33501, 65101, 66203, 1000003])
def test_sums_are_those_of_the_unfused_deposit(precision, n, k):
    import torch
    npart = k + 5003
    pos = _line(n, npart, k, precision, k)
    sums = []
    for flags in (nupm.PM_UNFUSED_DEPOSIT, nupm.PM_KEEP_DEPOSIT):
        pm = nupm.PM(n, npart, float(n), 0.3, 0.0, n_kbins=8, precision=precision, flags=flags)
        pm.deposit(pos)
        sums.append(pm.field(nupm.FIELD_DEPOSIT))
        pm.check()
        pm.close()
    assert torch.equal(*sums)


@pytest.mark.parametrize("k,wraps", [(65535, False), (70000, True)])
def test_a_wrapped_sum_of_a_shared_row_is_reported(k, wraps):
    import torch
    pos = torch.zeros((6, k), dtype=torch.int32, device="cuda")
    pos[0] = 77
    pm = nupm.PM(512, k, 512.0, 0.3, 0.0, n_kbins=8, precision="fp32")
    pm.deposit(pos)
    if wraps:
        with pytest.raises(nupm.PMError):
            pm.check()
    else:
        pm.check()
    pm.close()


def test_one_long_row_does_not_hold_up_the_grid():
    npart, ms = 2 ** 24, []
    pm = nupm.PM(512, npart, 512.0, 0.3, 0.0, n_kbins=8, precision="fp32")
    for k in (0, npart // 5):
        pos = _line(512, npart, k, "fp32", 3)
        best = float("inf")
        for _ in range(5):
            pm.timing(True)
            pm.deposit(pos)
            best = min(best, pm.get_timing()["fft_x_fwd"][0])
        ms.append(best)
    pm.check()
    pm.close()
    assert ms[1] < 35.0 * ms[0], ms     # 48 times as long by one warp a row, 22 shared
