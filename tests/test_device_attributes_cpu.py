"""Dynamic shared memory above 48 KB is allowed per device: a second device of
the process launches every kernel that the first one did.  The host code runs
against a recording CUDA runtime (no GPU)."""
import ctypes as C

import pytest

from fake_cuda import Fake
from paper_1209_0461_gb300 import nupm


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return Fake(tmp_path_factory.mktemp("fake"))


def _kick(fake, ctx, tuning):
    L, buf = fake.L, C.create_string_buffer(8 * 64)
    t = (C.c_int32 * 4)(*tuning)
    for rc in (L.pm_set_tuning(ctx, t), L.pm_deposit(ctx, buf), L.pm_nu_response(ctx, 0.1, None, None, 0, None, None, None, None),
               L.pm_kick(ctx, buf, buf, 0.1, 0.5, None)):
        assert rc == nupm.PM_OK, L.pm_last_error(ctx)


@pytest.mark.parametrize("precision", [nupm.PM_FP32, nupm.PM_FP64])
@pytest.mark.parametrize("n,flags,tuning", [
    (64, 0, (0, 0, 16, 2)), (192, 0, (-1, -1, 16, 0)), (192, 0, (1, 1, 16, 2)), (256, 0, (0, 0, 16, 2)),
    (512, 0, (1, 2, 16, 2)), (1024, 0, (-1, -1, 16, 2)), (256, nupm.PM_SPECTRAL_GRADIENT, (0, 2, 16, 0)), (256, nupm.PM_FUSED_GATHER, (1, 1, 16, 0)),
    (256, nupm.PM_TMA_COLUMNS, (0, 0, 16, 0)), (256, nupm.PM_UNFUSED_DEPOSIT, (1, 1, 16, 0))])
def test_second_device_launches_what_the_first_did(fake, precision, n, flags, tuning):
    runs = []
    for device in (0, 1):
        fake.L.fake_set_device(device)
        fake.clear()
        ctx = fake.init(n, precision=precision, flags=flags)
        _kick(fake, ctx, tuning)
        runs.append(fake.log())
        fake.L.pm_free(ctx)
    fake.L.fake_set_device(0)
    assert all(kind != "bad" for kind, _ in runs[0] + runs[1])
    assert runs[0] == runs[1] and len(runs[0]) > 12


def test_second_device_batch(fake):
    for device in (0, 1):
        fake.L.fake_set_device(device)
        fake.clear()
        ctx = [fake.init(192, n_kbins=16) for _ in range(2)]
        arr, out, buf = (C.c_void_p * 2)(*[c.value for c in ctx]), C.c_void_p(), C.create_string_buffer(8 * 64)
        assert fake.L.pm_batch_create(arr, 2, None, C.byref(out)) == nupm.PM_OK
        p = (C.c_void_p * 2)(*[C.addressof(buf)] * 2)
        a, k = (C.c_double * 2)(0.1, 0.1), (C.c_double * 2)(0.5, 0.5)
        assert fake.L.pm_batch_kick(out, p, p, a, k, None, None, None) == nupm.PM_OK, fake.L.pm_batch_last_error(out)
        assert all(kind != "bad" for kind, _ in fake.log())
        fake.L.pm_batch_free(out)
        for c in ctx:
            fake.L.pm_free(c)
    fake.L.fake_set_device(0)
