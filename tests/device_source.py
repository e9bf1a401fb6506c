"""Device functions of the CUDA sources compiled for the host: the text of the
named functions with the few intrinsics that they call, undefined behaviour of
C++ trapped."""
import ctypes as C
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1209_0461_gb300", "csrc")

SHIMS = r"""
#include <math.h>
#include <stdint.h>
#include <string.h>
#define __device__
#define __forceinline__ inline
struct CellSize { double d, fd_scale; float fd_scale_f; unsigned long long rm; int re; };
static inline long long __double_as_longlong(double x) { long long b; memcpy(&b, &x, 8); return b; }
static inline double __hiloint2double(int hi, int lo) {
  unsigned long long b = ((unsigned long long)(unsigned)hi << 32) | (unsigned)lo; double x; memcpy(&x, &b, 8); return x; }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
  return (unsigned long long)(((unsigned __int128)a * b) >> 64); }
static inline int __clz(unsigned u) { return u ? __builtin_clz(u) : 32; }
static inline unsigned __funnelshift_lc(unsigned lo, unsigned hi, unsigned s) {
  return s >= 32 ? lo : s ? hi << s | lo >> (32 - s) : hi; }
"""


def function_text(source, name):
    """The definition of a __device__ function of a source file."""
    text = open(os.path.join(CSRC, source)).read()
    m = re.search(r"^__device__[^\n;]*\b%s\(" % name, text, re.M)
    end = text.index("\n}\n", m.start())
    return text[m.start():end + 3]


def compile_host(out_dir, source, names, wrappers):
    src = os.path.join(str(out_dir), "host.cpp")
    with open(src, "w") as f:
        f.write(SHIMS + "".join(function_text(source, n) for n in names) + 'extern "C" {\n' + wrappers + "}\n")
    so = os.path.join(str(out_dir), "host.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-std=c++17", "-fsanitize=undefined",
                    "-fsanitize-undefined-trap-on-error", "-fno-sanitize=signed-integer-overflow", "-o", so, src], check=True)
    return C.CDLL(so)
