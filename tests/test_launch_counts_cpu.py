"""The launch counts that pm_get_timing reports are the kernels launched, stage
by stage summed over a kick, on both sides of each rule that adds or drops a
launch.  The host code runs against a recording CUDA runtime (no GPU)."""
import ctypes as C

import numpy as np
import pytest

from fake_cuda import Fake
from paper_1209_0461_gb300 import nupm


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return Fake(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("prepare", [False, True])
@pytest.mark.parametrize("n,precision,nk,nh,m_nu,rows", [
    (64, nupm.PM_FP32, 32, 63, 0.3, 0), (64, nupm.PM_FP64, 32, 64, 0.3, 0), (128, nupm.PM_FP32, 9, 227, 0.3, 1),
    (128, nupm.PM_FP64, 9, 228, 0.3, 2), (192, nupm.PM_FP32, 8, 0, 0.3, 2), (256, nupm.PM_FP32, 256, 8, 0.3, 2),
    (256, nupm.PM_FP32, 256, 128, 0.0, 0), (1024, nupm.PM_FP32, 256, 8, 0.3, 0), (1024, nupm.PM_FP32, 300, 4, 0.3, 0)])
def test_reported_launches_are_the_launches(fake, n, precision, nk, nh, m_nu, rows, prepare):
    L, buf = fake.L, C.create_string_buffer(8 * 64)
    ctx = fake.init(n, precision=precision, n_kbins=nk, m_nu=m_nu, n_hist_max=max(nh, 1))
    assert L.pm_set_tuning(ctx, (C.c_int32 * 4)(-1, -1, 16, rows)) == nupm.PM_OK
    ah = np.linspace(0.02, 0.05, max(nh, 1))
    a_hist = ah.ctypes.data_as(C.POINTER(C.c_double)) if nh else None
    hist = np.ones((max(nh, 1), nk))
    hp = hist.ctypes.data if nh else None
    assert L.pm_timing(ctx, 1) == nupm.PM_OK
    fake.clear()
    if prepare:
        assert L.pm_nu_prepare(ctx, 0.1, a_hist, hp, nh) == nupm.PM_OK
    assert L.pm_deposit(ctx, buf) == nupm.PM_OK
    assert L.pm_nu_response(ctx, 0.1, a_hist, hp, nh, None, None, None, None) == nupm.PM_OK
    assert L.pm_kick(ctx, buf, buf, 0.1, 0.5, None) == nupm.PM_OK
    log = fake.log()
    launches = np.zeros(len(nupm.STAGES), np.int64)
    assert L.pm_get_timing(ctx, None, launches.ctypes.data_as(C.POINTER(C.c_int64)), None) == nupm.PM_OK
    names = [what for kind, what in log if kind == "run"]
    assert launches.sum() == len(names), (dict(zip(nupm.STAGES, launches)), names)
    resp = [x for x in names if "k_nu_" in x or "k_fac_table" in x or "k_green_table" in x]
    assert launches[nupm.STAGES.index("response")] == len(resp), resp
    assert any("k_nu_nodes" in x for x in names) == (m_nu > 0 and nk * nh >= 2048)
    L.pm_free(ctx)
