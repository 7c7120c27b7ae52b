"""FP32 magnitudes behind the column bounds of the tensor-core Gram (csrc/gramnum.cuh), compiled for the host:
a bound that is not flagged as out of range has the FP64 bound's value to 2^-19, or both lie below 2^-102,
where every exponent is clamped alike."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = r"""
#include "gramnum.cuh"
extern "C" void run(long n, const double* lo, const double* hi, const double* lam, float* bound, unsigned char* out) {
  for (long i = 0; i < n; ++i) {
    bool o = false;
    float w = 1.f;
    for (int k = 0; k < 3; ++k) w *= (float)lam[3 * i + k];
    td::tc_weight32(w, o);
    bound[i] = (td::tc_abs32(lo[i], o) + td::tc_abs32(hi[i], o)) * w;
    out[i] = o;
  }
}
"""


@pytest.mark.parametrize("smallest", [1.0, 1e-12, 1e-13, 1e-20, 1e-40, 1e-60])
def test_bounds_are_right_or_flagged(tmp_path, smallest):
    src, lib = str(tmp_path / "t.cpp"), str(tmp_path / "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(HERE, "..", "paper_2310_10722_gb300", "csrc"), src, "-o", lib], check=True)
    rng = np.random.default_rng(11)
    n = 200000
    lo, hi = rng.choice([-1.0, 1.0], (2, n)) * np.exp2(rng.uniform(-130.0, 102.0, (2, n)))
    lam = np.exp(rng.uniform(np.log(smallest), 0.0, (n, 3)))
    lam[: n // 4] = smallest                                  # every weight at its smallest
    bound, out = np.empty(n, dtype=np.float32), np.empty(n, dtype=np.uint8)
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
    ctypes.CDLL(lib).run(ctypes.c_long(n), ptr(lo), ptr(hi), ptr(lam), ptr(bound), ptr(out))
    want = (np.abs(lo) + np.abs(hi)) * lam.prod(axis=1)
    right = (np.abs(bound - want) <= want * 2.0 ** -19) | ((want < 2.0 ** -102) & (bound < 2.0 ** -102))
    assert (right | (out != 0)).all()
    # values within FP32's range and weights of at most the default cutoff's size need no second pass
    if smallest >= 1e-12:
        assert not out[np.maximum(np.abs(lo), np.abs(hi)) < 2.0 ** 99].any()
