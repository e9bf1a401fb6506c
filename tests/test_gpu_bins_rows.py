"""Power sums with the lane's mode count fixed at compile time: every grid size
that takes that path in either precision, one bin, more bins than the fused
form holds, and ragged counts, against the oracle's bins of the same spectrum."""
import numpy as np
import pytest

from oracle import pm_oracle as O
from paper_1209_0461_gb300 import nupm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,n,nk", [("fp64", 16, 3), ("fp64", 32, 40), ("fp64", 64, 1), ("fp64", 64, 300),
                                            ("fp64", 128, 33), ("fp64", 192, 64), ("fp64", 256, 17),
                                            ("fp32", 32, 5), ("fp32", 64, 64), ("fp32", 192, 1), ("fp32", 192, 300)])
def test_bins_of_the_spectrum(precision, n, nk):
    import torch
    npart = 4 * n * n + 3
    rng = np.random.default_rng(n + nk)
    pos = rng.random((3, npart)) * 50.0
    pm = nupm.PM(n, npart, 50.0, 0.3, 0.0, n_kbins=nk, precision=precision)
    if precision == "fp64":
        p = torch.from_numpy(pos).cuda()
    else:
        u = pos / (50.0 / n)
        off = np.minimum((u - np.floor(u)).astype(np.float32), np.float32(1 - 2.0 ** -24))
        p = torch.from_numpy(np.concatenate([np.floor(u).astype(np.int32), off.view(np.int32)])).cuda()
    pm.deposit(p)
    spec = pm.field(nupm.FIELD_DELTA_K).cpu().numpy().astype(np.complex128)
    cnt, ks, ps = pm.bins()
    pm.deposit(p)
    again = pm.bins()[2]
    pm.check()
    pm.close()
    ref = O.bin_power(spec, 50.0, nk)
    c, s = ref["count"], ref["psum"]
    assert np.array_equal(cnt, c)
    # FP64: sums of up to 1e7 terms in another order; FP32: 2^-24 a mode, float-pair accumulators
    np.testing.assert_allclose(ps, s, rtol=1e-10 if precision == "fp64" else 2e-6)
    assert np.array_equal(ps, again)
