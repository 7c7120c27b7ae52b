// FP32 magnitudes for the column bounds of the tensor-core Gram (absorb.cu), on bit patterns: usable on the
// host too, where the tests run them.  The bound of a value v with row weight w is tc_abs32(v) * w; where
// `out` stays false it is within 2^-19 of the FP64 product, or both are below 2^-102.
#pragma once

#include "ieee.cuh"

namespace td {

// |x| as an FP32 value truncated from the bit pattern (no FP64 instruction); out: x is beyond 2^100.
TD_IEEE_HD float tc_abs32(double x, bool& out) {
  const uint64_t u = ieee_bits(x);
  const uint32_t hi = (uint32_t)(u >> 32) & 0x7FFFFFFFu, lo = (uint32_t)u;
  out |= hi >= (1023u + 100u) << 20;
  return hi < (1023u - 126u) << 20 ? 0.f : ieee_float(((hi - (896u << 20)) << 3) | (lo >> 29));
}
TD_IEEE_HD float tc_abs32(float x, bool& out) {
  out |= !(fabsf(x) < 1.2676506e30f);
  return fabsf(x);
}

// out: the product w of the FP32 bond weights (each in (0, 1], so no factor undoes an earlier underflow)
// is subnormal or zero: the row would leave the bound although its values may not be small.
TD_IEEE_HD void tc_weight32(float w, bool& out) { out |= !(w >= 1.17549435e-38f); }

}  // namespace td
