"""A row sort that stops between its count and its scan (a launch that fails,
as the first use of a kernel on a full device does): no scatter by stale
cursors, and the counts are cleared before the next count, so that the retry
sorts as if nothing had happened.  The host code runs against a recording CUDA
runtime (no GPU)."""
import ctypes as C

import pytest

from fake_cuda import Fake
from paper_1209_0461_gb300 import nupm


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    return Fake(tmp_path_factory.mktemp("fake"))


def _names(log, part):
    return [i for i, (kind, what) in enumerate(log) if kind != "set" and part in what]


@pytest.mark.parametrize("precision", [nupm.PM_FP32, nupm.PM_FP64])
@pytest.mark.parametrize("n,scan", [(64, "k_scan_one"), (128, "k_scan_blocks"), (128, "k_scan_totals"), (128, "k_scan_add")])
def test_deposit_retried_after_a_failed_scan(fake, precision, n, scan):
    L, buf = fake.L, C.create_string_buffer(8 * 64)
    ctx = fake.init(n, precision=precision)
    assert L.pm_deposit(ctx, buf) == nupm.PM_OK
    fake.clear()
    L.fake_fail(scan.encode(), 1)
    assert L.pm_deposit(ctx, buf) == -4
    log = fake.log()
    bad = [i for i in _names(log, scan) if log[i][0] == "bad"]
    assert len(bad) == 1 and not [i for i in _names(log, "k_row_scatter") if i > bad[0]]
    assert L.pm_deposit(ctx, buf) == nupm.PM_OK
    log = fake.log()
    count = [i for i in _names(log, "k_row_count") if i > bad[0]][0]
    assert ("set", 4 * (n * n + 1)) in log[bad[0]:count]
    fake.clear()
    assert L.pm_deposit(ctx, buf) == nupm.PM_OK
    assert not [k for k in fake.log() if k[0] == "set"]          # an undisturbed sort clears nothing by itself
    L.pm_free(ctx)


@pytest.mark.parametrize("direct_first", [False, True])
def test_batch_retried_after_a_failed_scan(fake, direct_first):
    L, buf, n = fake.L, C.create_string_buffer(8 * 64), 64
    ctx = [fake.init(n) for _ in range(2)]
    arr, out = (C.c_void_p * 2)(*[c.value for c in ctx]), C.c_void_p()
    assert L.pm_batch_create(arr, 2, None, C.byref(out)) == nupm.PM_OK
    p = (C.c_void_p * 2)(*[C.addressof(buf)] * 2)
    a, k = (C.c_double * 2)(0.1, 0.1), (C.c_double * 2)(0.5, 0.5)

    def kick():
        return L.pm_batch_kick(out, p, p, a, k, None, None, None)

    assert kick() == nupm.PM_OK
    fake.clear()
    if direct_first:                                     # a direct sort of one box fails, the batch follows
        L.fake_fail(b"k_scan_one", 1)
        assert L.pm_deposit(ctx[1], buf) == -4
        want = 1
    else:
        L.fake_fail(b"PScan", 1)
        assert kick() == -4
        want = 2
    log = fake.log()
    bad = [i for i, e in enumerate(log) if e[0] == "bad"]
    assert len(bad) == 1 and not [i for i in _names(log, "catter") if i > bad[0]]
    assert kick() == nupm.PM_OK
    log = fake.log()
    count = [i for i in _names(log, "PCount") if i > bad[0]][0]
    assert log[bad[0]:count].count(("set", 4 * (n * n + 1))) == want
    fake.clear()
    assert kick() == nupm.PM_OK and L.pm_deposit(ctx[0], buf) == nupm.PM_OK
    assert ("set", 4 * (n * n + 1)) not in fake.log()
    L.pm_batch_free(out)
    for c in ctx:
        L.pm_free(c)
