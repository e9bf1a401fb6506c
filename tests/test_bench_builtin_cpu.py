"""The benchmark's byte model knows which form of the bin sums runs, also where
the tuning is left to the library: compared with what the entry points launch
on a recording CUDA runtime (no GPU)."""
import ctypes as C

import pytest

import bench
from fake_cuda import Fake
from paper_1209_0461_gb300 import nupm, synth


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return Fake(tmp_path_factory.mktemp("fake"))


@pytest.mark.parametrize("n,precision,nk,spectral,tuning", [
    (1024, "fp32", 256, False, None), (1024, "fp32", 256, False, [0, -1, 4, 0]), (1024, "fp32", 257, False, None),
    (1024, "fp32", 256, True, None), (1024, "fp32", 256, True, [0, 2, 4, 0]), (1024, "fp32", 256, False, [0, 1, 4, 0]),
    (1024, "fp64", 256, False, None), (512, "fp32", 256, False, None), (512, "fp32", 256, False, [-1, 2, 4, 0]),
    (256, "fp32", 64, False, [1, -1, 4, 0])])
def test_bins_form_of_the_model_is_the_launched_one(fake, n, precision, nk, spectral, tuning):
    w = synth.with_(synth.WORKLOADS["pm1024_p512_fp32"], ngrid=n, precision=precision, n_kbins=nk)
    ctx = fake.init(n, precision=nupm.PM_FP32 if precision == "fp32" else nupm.PM_FP64, n_kbins=nk,
                    flags=nupm.PM_SPECTRAL_GRADIENT if spectral else 0)
    if tuning:
        assert fake.L.pm_set_tuning(ctx, (C.c_int32 * 4)(*tuning)) == nupm.PM_OK
    fake.clear()
    assert fake.L.pm_deposit(ctx, C.create_string_buffer(64 * 8)) == nupm.PM_OK
    in_z = any("k_bin_plane0" in str(what) for _, what in fake.log())
    fake.L.pm_free(ctx)
    assert bench.bins_in_z(w, bench.effective_tuning(w, tuning, spectral)) == in_z
    # the model without that: a whole spectrum's read too many or too few
    assert (bench.stage_bytes(w, "bins", False, spectral, in_z) < 2 ** 25) == in_z
