"""The integer quotient and square root of the Jacobi angles (csrc/ieee.cuh), compiled for the host:
bit for bit IEEE 754's results (numpy's), from FP32 estimates that are off by up to a few units, as the
device's are."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = r"""
#include "ieee.cuh"
using namespace td;
static float off(float y, int k) { uint32_t u; std::memcpy(&u, &y, 4); u += k; std::memcpy(&y, &u, 4); return y > 1.f ? 1.f : y; }
extern "C" void run(long n, int k, const double* a, const double* b, double* q, double* s, long* bad) {
  *bad = 0;
  for (long i = 0; i < n; ++i) {
    q[i] = ieee_div(a[i], b[i]);
    s[i] = ieee_sqrt(a[i]);
    // the significands with an estimate k units off: the same integers
    const uint64_t B = (ieee_bits(b[i]) & kIeeeFrac) | kIeeeOne;
    uint64_t A = (ieee_bits(a[i]) & kIeeeFrac) | kIeeeOne;
    const uint64_t V = A << (i & 1);
    A <<= A < B;
    const float bf = ieee_float(0x3F800000u | (uint32_t)((B >> 29) & 0x7FFFFFu));
    const float vf = ieee_float((uint32_t)(((127 + (i & 1)) << 23) | (int)((ieee_bits(a[i]) >> 29) & 0x7FFFFFu)));
    *bad += ieee_div_sig(A, B, off(1.f / bf, k)) != ieee_div_sig(A, B, 1.f / bf);
    *bad += ieee_sqrt_sig(V, off(1.f / std::sqrt(vf), k)) != ieee_sqrt_sig(V, 1.f / std::sqrt(vf));
  }
}
"""


@pytest.mark.parametrize("kind", ["random", "near-one", "few-bits", "all-exponents", "special"])
def test_quotient_and_root_are_ieee(tmp_path, kind):
    src, lib = str(tmp_path / "t.cpp"), str(tmp_path / "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(HERE, "..", "paper_2310_10722_gb300", "csrc"), src, "-o", lib], check=True)
    run = ctypes.CDLL(lib).run
    rng = np.random.default_rng(7)
    n = 200000
    frac = rng.integers(0, 1 << 52, size=(2, n), dtype=np.uint64)
    ex = rng.integers(990, 1060, size=(2, n), dtype=np.uint64)
    if kind == "near-one":      # significands next to 1 and 2
        frac = np.where(rng.random((2, n)) < 0.5, frac % 64, (1 << 52) - 1 - frac % 64).astype(np.uint64)
    elif kind == "few-bits":
        frac &= ~((np.uint64(1) << rng.integers(20, 52, size=(2, n), dtype=np.uint64)) - np.uint64(1))
    elif kind == "all-exponents":
        ex = rng.integers(0, 2048, size=(2, n), dtype=np.uint64)
    a, b = ((ex << np.uint64(52)) | frac).view(np.float64)
    if kind == "special":
        v = np.array([0.0, 1.0, 2.0, np.inf, np.nan, 5e-324, 2.0 ** -1022, np.finfo(float).max, 3.0, 2.0 ** -1074 * 3])
        a, b = (x.ravel().copy() for x in np.meshgrid(v, v))
    sign = np.where(np.arange(a.size) % 3 == 0, -1.0, 1.0)
    b = b * sign
    q, s, bad = np.empty_like(a), np.empty_like(a), ctypes.c_long()
    ptr = lambda x: x.ctypes.data_as(ctypes.c_void_p)
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    for k in (-3, 0, 3):
        run(ctypes.c_long(a.size), ctypes.c_int(k), ptr(a), ptr(b), ptr(q), ptr(s), ctypes.byref(bad))
        assert bad.value == 0
    with np.errstate(all="ignore"):
        for got, want in ((q, a / b), (s, np.sqrt(a))):
            same = (got.view(np.uint64) == want.view(np.uint64)) | (np.isnan(got) & np.isnan(want))
            assert same.all(), (a[~same][:3], b[~same][:3])
