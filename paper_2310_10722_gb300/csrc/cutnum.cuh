// FP32 numbers of the cuts (cut.cuh), on bit patterns: usable on the host too, where the tests run them.
#pragma once

#include "ieee.cuh"

namespace td {

// FP32 value of x 2^-E, truncated to 24 bits, from the bit pattern (integer pipes only; below the
// FP32 normal range: 0).
TD_IEEE_HD float cut_f32(double x, int E) {
  const uint64_t u = ieee_bits(x);
  const uint32_t hi = (uint32_t)(u >> 32), lo = (uint32_t)u;
  const int e = (int)((hi >> 20) & 0x7FFu) - 1023 - E + 127;
  if (e <= 0) return 0.0f;
  return ieee_float((hi & 0x80000000u) | ((uint32_t)e << 23) | ((hi & 0xFFFFFu) << 3) | (lo >> 29));
}

// |e| sqrt(theta_j / theta_0) as a bit pattern, which orders the residuals -- infinity and NaN above all
// finite ones, so a residual that is not a number fails the test that it is small.  The thetas (squared
// singular values of a matrix of magnitude 2^expo) are scaled by 2^(-2 expo): unscaled they leave FP32's range
// beyond |expo| = 63, and zero times infinity read as no residual at all.
TD_IEEE_HD uint32_t cut_residual(float e, double theta_j, double theta_0, int expo) {
  const float r = fabsf(e) * sqrtf(cut_f32(theta_j, 2 * expo) / cut_f32(theta_0, 2 * expo));
  return ieee_float_bits(r) & 0x7FFFFFFFu;
}

}  // namespace td
