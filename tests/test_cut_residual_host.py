"""The residual by which a cut accepts its vectors (csrc/cutnum.cuh), compiled for the host: right over the
whole range of magnitudes that the cuts admit, and never small when it is not a number."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
SRC = r"""
#include "cutnum.cuh"
extern "C" void run(long n, const float* e, const double* tj, const double* t0, const int* ex, float* r) {
  for (long i = 0; i < n; ++i) r[i] = td::ieee_float(td::cut_residual(e[i], tj[i], t0[i], ex[i]));
}
"""


@pytest.fixture(scope="module")
def residual(tmp_path_factory):
    at = tmp_path_factory.mktemp("residual")
    src, lib = str(at / "t.cpp"), str(at / "t.so")
    with open(src, "w") as f:
        f.write(SRC)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(HERE, "..", "paper_2310_10722_gb300", "csrc"), src, "-o", lib], check=True)
    fn = ctypes.CDLL(lib).run

    def call(e, tj, t0, ex):
        e, tj, t0, ex = (np.ascontiguousarray(a, dtype=t) for a, t in zip(np.broadcast_arrays(e, tj, t0, ex), ("f4", "f8", "f8", "i4")))
        r = np.empty(e.shape, dtype=np.float32)
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        fn(ctypes.c_long(e.size), ptr(e), ptr(tj), ptr(t0), ptr(ex), ptr(r))
        return r
    return call


def test_right_at_every_magnitude(residual):
    rng = np.random.default_rng(3)
    ex = np.repeat(np.arange(-399, 400), 64)
    t0 = np.exp2(2.0 * ex + rng.uniform(0.0, 22.0, ex.size))       # sigma_1^2: up to 2048 x 1024 entries
    tj = t0 * np.exp2(rng.uniform(-34.0, 0.0, ex.size))            # sigma_k >= 1e-5 sigma_1
    e = np.exp2(rng.uniform(-56.0, -6.0, ex.size)).astype(np.float32)
    want = e * np.sqrt(tj / t0)
    # two values truncated to 24 bits (2^-23 each, halved by the root) and three FP32 roundings
    assert (np.abs(residual(e, tj, t0, ex) / want - 1) < 2.5 * 2.0 ** -23).all()


@pytest.mark.parametrize("ex", [-399, -75, 0, 75, 399])
def test_not_a_number_is_not_small(residual, ex):
    unit = 4.0 ** ex
    for e, tj, t0 in ((np.nan, unit, unit), (-np.nan, unit, unit), (np.inf, unit, unit), (1e-9, unit, 0.0), (0.0, 0.0, 0.0)):
        assert not residual(e, tj, t0, ex)[()] <= 1e-2
