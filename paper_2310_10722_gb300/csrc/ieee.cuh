// FP64 quotient and square root, rounded to nearest, in integer arithmetic.
//
// Why: a warp's FP64 instruction takes the SM 19 cycles on this chip and its own scheduler 64, an
// integer one 0.25 and 1 -- a division is 7 and a square root 10 FP64 instructions, and the angles of the
// Jacobi rotations are a chain of two divisions and a square root.  Here each takes ~60 integer instructions
// and none in FP64.  Measured (core time of a decode): rotated d9 chi 8, 1000 shots 129.0 -> 121.5 ms, its FP64 152
// shots 47.4 -> 43.5, rotated d7 FP64, 48 shots 18.9 -> 16.7, rotated d5, 37 shots 7.37 -> 6.80; the sweep of
// rotated d9 chi 16, 16 shots 128 -> 123 ms, a gradient 185 -> 179 ms.  Both are correctly rounded, as
// IEEE 754 defines the operations, so the values are those of `/` and sqrt() bit for bit.
//
// How: Newton's iteration from an FP32 estimate (relative error below 2^-21), one cubic step in fixed
// point (1 / (1 - e) = 1 + e + e^2 + O(e^3), (1 - e)^(-1/2) = 1 + e / 2 + 3 e^2 / 8 + O(e^3)), which leaves an error below
// 2^-58, and the integer nearest to the scaled result from its exact remainder modulo 2^64: for a quotient
// r of the significands, A 2^52 - r B; for a root, V 2^52 - r^2.  Neither can lie midway between two
// 53-bit values.  Operands or results that are zero, subnormal, infinite or NaN take the FP64 operation.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

namespace td {

#ifdef __CUDA_ARCH__
#define TD_IEEE_HD __device__ __forceinline__
TD_IEEE_HD uint64_t ieee_bits(double x) { return (uint64_t)__double_as_longlong(x); }
TD_IEEE_HD double ieee_value(uint64_t u) { return __longlong_as_double((long long)u); }
TD_IEEE_HD uint64_t ieee_mulhi(uint64_t a, uint64_t b) { return __umul64hi(a, b); }
TD_IEEE_HD int64_t ieee_mulhi_s(int64_t a, int64_t b) { return __mul64hi(a, b); }
TD_IEEE_HD float ieee_float(uint32_t u) { return __uint_as_float(u); }
TD_IEEE_HD uint32_t ieee_float_bits(float x) { return __float_as_uint(x); }
TD_IEEE_HD float ieee_rcp_est(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
TD_IEEE_HD float ieee_rsqrt_est(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
#else
#define TD_IEEE_HD inline
TD_IEEE_HD uint64_t ieee_bits(double x) { uint64_t u; std::memcpy(&u, &x, 8); return u; }
TD_IEEE_HD double ieee_value(uint64_t u) { double x; std::memcpy(&x, &u, 8); return x; }
TD_IEEE_HD uint64_t ieee_mulhi(uint64_t a, uint64_t b) { return (uint64_t)((unsigned __int128)a * b >> 64); }
TD_IEEE_HD int64_t ieee_mulhi_s(int64_t a, int64_t b) { return (int64_t)((__int128)a * b >> 64); }
TD_IEEE_HD float ieee_float(uint32_t u) { float x; std::memcpy(&x, &u, 4); return x; }
TD_IEEE_HD uint32_t ieee_float_bits(float x) { uint32_t u; std::memcpy(&u, &x, 4); return u; }
TD_IEEE_HD float ieee_rcp_est(float x) { return 1.0f / x; }
TD_IEEE_HD float ieee_rsqrt_est(float x) { return 1.0f / std::sqrt(x); }
#endif

constexpr uint64_t kIeeeOne = 1ull << 52, kIeeeFrac = kIeeeOne - 1;

// round(A 2^52 / B) for significands A, B in [2^52, 2^54), [2^52, 2^53) with 1 <= A / B < 2; y0: an
// estimate of 2^52 / B.
TD_IEEE_HD uint64_t ieee_div_sig(uint64_t A, uint64_t B, float y0) {
  const uint32_t Y = (uint32_t)(y0 * 2147483648.0f);              // 2^31 y0, y0 in (1/2, 1]
  const int64_t E = -(int64_t)(B * Y);                            // 2^83 e, e = 1 - b y0 (mod 2^64)
  const int32_t Eh = (int32_t)(E >> 32);
  const int64_t F = E + (((int64_t)Eh * Eh) >> 19);               // 2^83 (e + e^2)
  const int64_t hi = (int64_t)(int32_t)(F >> 32) * (int64_t)Y;
  const int64_t lo = (int64_t)(((uint64_t)(uint32_t)F * Y) >> 32);
  const uint64_t X = ((uint64_t)Y << 32) + (uint64_t)((hi + lo) >> 19);   // 2^63 / b
  uint64_t r = ieee_mulhi(A << 1, X);
  const int64_t rem = (int64_t)((A << 52) - r * B);               // in (-B / 2, 3 B / 2)
  if (2 * rem > (int64_t)B) ++r;
  return r;
}

// round(sqrt(V 2^52)) for V in [2^52, 2^54); y0: an estimate of sqrt(2^52 / V).
TD_IEEE_HD uint64_t ieee_sqrt_sig(uint64_t V, float y0) {
  const uint32_t Y = (uint32_t)(y0 * 2147483648.0f);              // 2^31 y0, y0 in (1/2, 1]
  const uint64_t V10 = V << 10;
  const int64_t E = (int64_t)((1ull << 60) - ieee_mulhi(V10, (uint64_t)Y * Y));   // 2^60 e, e = 1 - v y0^2
  const int64_t Eh = E >> 20;
  const int64_t H = (E >> 1) + ((3 * Eh * Eh) >> 23);             // 2^60 (e / 2 + 3 e^2 / 8)
  const uint64_t T = (V10 >> 32) * Y + (((V10 & 0xFFFFFFFFull) * Y) >> 32);   // 2^61 v y0
  uint64_t r = (T + (uint64_t)(ieee_mulhi_s((int64_t)T, H << 24) >> 20)) >> 9;
  const int64_t rem = (int64_t)((V << 52) - r * r);               // in (-r, 3 r)
  if (rem > (int64_t)r) ++r;
  return r;
}

// a / b
TD_IEEE_HD double ieee_div(double a, double b) {
  const uint64_t ua = ieee_bits(a), ub = ieee_bits(b);
  const int ea = (int)(ua >> 52) & 0x7FF, eb = (int)(ub >> 52) & 0x7FF;
  uint64_t A = (ua & kIeeeFrac) | kIeeeOne;
  const uint64_t B = (ub & kIeeeFrac) | kIeeeOne;
  int e = ea - eb + 1023;
  if (A < B) {
    A <<= 1;
    --e;
  }
  if (ea == 0 || ea == 0x7FF || eb == 0 || eb == 0x7FF || e < 1 || e > 2045) return a / b;
  const uint64_t r = ieee_div_sig(A, B, ieee_rcp_est(ieee_float(0x3F800000u | (uint32_t)((B >> 29) & 0x7FFFFFu))));
  return ieee_value(((ua ^ ub) & 0x8000000000000000ull) | (((uint64_t)e << 52) + (r - kIeeeOne)));
}

// sqrt(x)
TD_IEEE_HD double ieee_sqrt(double x) {
  const uint64_t u = ieee_bits(x);
  const int ex = (int)(u >> 52);   // with the sign
  if (ex < 1 || ex >= 0x7FF) return sqrt(x);
  const int odd = (ex & 1) ^ 1;    // an odd power of two
  const uint64_t V = ((u & kIeeeFrac) | kIeeeOne) << odd;
  // the estimate's operand: V's upper bits as an FP32 value in [1, 4)
  const float v = ieee_float((uint32_t)(((127 + odd) << 23) | (int)((u >> 29) & 0x7FFFFFu)));
  const uint64_t r = ieee_sqrt_sig(V, ieee_rsqrt_est(v));
  return ieee_value(((uint64_t)((ex - 1023 - odd) / 2 + 1023) << 52) + (r - kIeeeOne));
}

TD_IEEE_HD float ieee_div(float a, float b) { return a / b; }
TD_IEEE_HD float ieee_sqrt(float x) { return sqrtf(x); }

}  // namespace td
