"""The FP64 stencil weights built from their bits: exact for every weight, zero
among them, without undefined behaviour of C++ (the host build traps on it)."""
import ctypes as C

import numpy as np
import pytest

from device_source import compile_host

WRAP = r"""
void powers(const unsigned* u, long n, int sh, int neg, double* out) {
  for (long i = 0; i < n; ++i) out[i] = exact_pow2(u[i], sh, neg != 0);
}
void products(const unsigned* a, const unsigned* b, long n, double* out) {
  for (long i = 0; i < n; ++i) out[i] = exact_product(a[i], b[i]);
}
"""


@pytest.fixture(scope="module")
def bits(tmp_path_factory):
    return compile_host(tmp_path_factory.mktemp("bits"), "grid_kernels.cuh", ["exact_pow2", "exact_product"], WRAP)


@pytest.mark.parametrize("sh,neg", [(16, 0), (16, 1), (13, 0), (13, 1), (32, 0)])
def test_powers(bits, sh, neg):
    g = np.random.default_rng(sh)
    u = np.concatenate([np.arange(70000), g.integers(0, 1 << 32, 50000), 2 ** np.arange(32, dtype=np.int64),
                        [0xffffffff]]).astype(np.uint32)
    out = np.empty(u.size)
    bits.powers(u.ctypes.data_as(C.c_void_p), C.c_long(u.size), sh, neg, out.ctypes.data_as(C.c_void_p))
    assert np.array_equal(out, (-1.0 if neg else 1.0) * u * 2.0 ** -sh)


def test_products(bits):
    g = np.random.default_rng(3)
    a = np.concatenate([[0, 65536, 0, 65536, 1, 65535], g.integers(0, 65537, 100000)]).astype(np.uint32)
    b = np.concatenate([[0, 65536, 65536, 0, 65536, 65535], g.integers(0, 65537, 100000)]).astype(np.uint32)
    out = np.empty(a.size)
    bits.products(a.ctypes.data_as(C.c_void_p), b.ctypes.data_as(C.c_void_p), C.c_long(a.size), out.ctypes.data_as(C.c_void_p))
    assert np.array_equal(out, a.astype(np.float64) * b * 2.0 ** -32)
