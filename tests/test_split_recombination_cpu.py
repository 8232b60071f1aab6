"""The recombination of the split product, compiled for the CPU from the kernel's own
source: the six level sums of one element against their exact integer sum, over
the whole range that each level can reach with 16, 32 and 64 products, and the
conversion to a double against the correctly rounded value.
"""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = os.path.join(ROOT, "paper_2602_05255_gb300", "csrc", "refresh_oz.cu")
SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
static inline int __float_as_int(float x) { int i; memcpy(&i, &x, 4); return i; }
static inline float __fmaf_rn(float a, float b, float c) { return fmaf(a, b, c); }
static inline int __float2int_rn(float x) { return (int)lrintf(x); }
static inline int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
static inline double __hiloint2double(int h, int l) {
    uint64_t b = ((uint64_t)(uint32_t)h << 32) | (uint32_t)l; double d; memcpy(&d, &b, 8); return d;
}
"""
MAIN = r"""
extern "C" void recombine(const float* a, int one_step, int e, long long* F, double* d) {
    int hi; uint32_t lo;
    oz_sum2(a[0], a[1], hi);
    oz_sum4(a[2], a[3], hi, lo);
    if (one_step) oz_sum6<true>(a[4], a[5], hi, lo);
    else oz_sum6<false>(a[4], a[5], hi, lo);
    *F = ((long long)hi << 32) | lo;
    *d = oz_to_double(hi, lo, e);
}
extern "C" double to_double(long long F, int e) { return oz_to_double((int)(F >> 32), (uint32_t)F, e); }
"""
BOUND = [256] + [128] * 6   # largest digits
SCALE = [-16, -24, -32, -40, -48, -56]   # the units of the levels 2 .. 6 and of the tail


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    text = open(SRC).read()
    parts = []
    for name in ("oz_sum2", "oz_sum4", "oz_sum6", "oz_to_double"):
        m = re.search(r"(?:template <[^>]*>\n)?__device__ __forceinline__ \w+ " + name + r"\(.*?\n}\n", text, re.S)
        assert m, name
        parts.append(m.group(0))
    d = tmp_path_factory.mktemp("recombine")
    src, so = str(d / "r.cpp"), str(d / "r.so")
    open(src, "w").write(SHIM + "".join(parts) + MAIN)
    subprocess.run(["g++", "-O1", "-fwrapv", "-ffp-contract=off", "-shared", "-fPIC", "-o", so, src], check=True)
    lib = ctypes.CDLL(so)
    lib.to_double.restype = ctypes.c_double
    lib.to_double.argtypes = [ctypes.c_longlong, ctypes.c_int]
    return lib


def limits(products):
    """The largest |level sum| in units of its level, the tail's in units of 2^-56."""
    n = [products * sum(BOUND[t] * BOUND[lv - 2 - t] for t in range(7) if 0 <= lv - 2 - t < 7) for lv in range(2, 7)]
    tail = sum(products * sum(BOUND[t] * BOUND[lv - 2 - t] for t in range(7) if 0 <= lv - 2 - t < 7) / 256.0 ** (lv - 7)
               for lv in range(7, 11))
    return n + [int(tail)]


@pytest.mark.parametrize("products", [16, 32, 64])
def test_level_sums_are_added_exactly(lib, products):
    g = np.random.Generator(np.random.PCG64(products))
    lim = limits(products)
    assert all(x < 2 ** 23 for x in lim[:5])
    F, d = ctypes.c_longlong(), ctypes.c_double()
    for trial in range(4000):
        if trial < 64:      # every combination of the largest values
            N = [x if trial >> i & 1 else -x for i, x in enumerate(lim)]
        else:
            N = [int(g.integers(-x, x + 1)) for x in lim]
        a = np.array([np.ldexp(float(x), s) for x, s in zip(N, SCALE)], np.float32)
        assert all(int(np.ldexp(float(v), -s)) == x for v, x, s in zip(a, N, SCALE))   # 24 bits hold them
        lib.recombine(a.ctypes.data_as(ctypes.c_void_p), products == 16, 0, ctypes.byref(F), ctypes.byref(d))
        want = sum(x << (56 + s) for x, s in zip(N, SCALE))
        assert F.value == want, (N, F.value - want)


def test_conversion_rounds_to_nearest_even(lib):
    g = np.random.Generator(np.random.PCG64(3))
    for trial in range(6000):
        F = int(g.integers(-2 ** 62, 2 ** 62)) >> int(g.integers(0, 62))
        if trial % 3 == 0:              # a tie, or one beside it
            m = int(g.integers(2 ** 52, 2 ** 53))
            sh = int(g.integers(1, 9))
            F = (m << sh) + (1 << (sh - 1)) + int(g.integers(-1, 2))
            F = -F if trial % 2 else F
        e = int(g.integers(-400, 400))
        assert lib.to_double(F, e) == np.ldexp(float(F), e - 56), (F, e)   # int to float rounds to even
    assert lib.to_double(2 ** 62 - 1, 0) == 64.0
    assert lib.to_double(0, 5) == 0.0
