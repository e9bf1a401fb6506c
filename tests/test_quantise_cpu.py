"""The integer quantisation of FP64 positions against the division that it
stands for, positions of both signs: every value that it decides is the
division's, and it decides negative ones as often as positive ones."""
import ctypes as C

import numpy as np
import pytest

from device_source import compile_host

WRAP = r"""
long run(const double* x, long n, double d, int* decided, long long* v) {
  CellSize cs; cs.d = d;
  const double r = 65536.0 / d; unsigned long long b; memcpy(&b, &r, 8);
  cs.rm = (b << 11) | (1ull << 63); cs.re = (int)(b >> 52);
  for (long i = 0; i < n; ++i) { Q q = 0; decided[i] = quant_fast(x[i], cs, q); v[i] = (long long)q; }
  return n;
}
"""


@pytest.fixture(scope="module")
def quant(tmp_path_factory):
    out = tmp_path_factory.mktemp("quant")
    import device_source
    value = "unsigned" if "unsigned& v)" in device_source.function_text("grid_kernels.cuh", "quant_fast") else "int"
    return compile_host(out, "grid_kernels.cuh", ["quant_fast"], WRAP.replace("Q q", value + " q"))


@pytest.mark.parametrize("d", [1.0, 100.0 / 32, 333.333 / 64, 7e-3 / 192, 1e6 / 128, 500.0 / 256, float(np.nextafter(2.0, 1))])
def test_decided_values_are_the_divisions(quant, d):
    g = np.random.default_rng(int(d * 1000) % 9973)
    k = g.integers(-(1 << 23), 1 << 23, 60000) * (d / 65536.0)             # weight boundaries and their neighbours
    x = np.concatenate([k, np.nextafter(k, np.inf), np.nextafter(k, -np.inf), (g.random(200000) - 0.5) * 64 * d,
                        np.sign(g.random(60000) - 0.5) * d * 10.0 ** g.uniform(-7, 5, 60000),
                        [0.0, -0.0, -1e-300, 5e-324, -5e-324, np.inf, -np.inf, np.nan, 1e300, -1e300]])
    dec, v = np.zeros(x.size, np.int32), np.zeros(x.size, np.int64)
    quant.run(x.ctypes.data_as(C.c_void_p), C.c_long(x.size), C.c_double(d), dec.ctypes.data_as(C.c_void_p),
              v.ctypes.data_as(C.c_void_p))
    dec = dec != 0
    u = x[dec] / d
    cf = np.floor(u)
    w = np.floor((u - cf) * 65536.0).astype(np.int64)
    assert np.array_equal(v[dec], cf.astype(np.int64) * 65536 + w)
    uni = slice(180000, 380000)                                              # even over [-32, 32) cells
    neg = x[uni] < 0
    assert dec[uni][neg].mean() > 0.999 and dec[uni][~neg].mean() > 0.999
