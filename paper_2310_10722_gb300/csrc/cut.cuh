// Truncation of one zip-up cut of the final contraction: the kept left singular vectors U of
// M (m x n) and the carry U^T M, from A = M^T (n x m, column-major, FP64), by one block.
//
// What bounds it: GB300 issues ~2 FP64 FMAs per clock and SM but 128 in FP32, so a cut costs what
// its FP64 operations cost.  A one-sided Jacobi SVD of the whole matrix spends ~90 m^3 of them
// where a cut keeps k << m vectors and, inside the kept space, any orthonormal basis will do (a
// rotation of it is a gauge of the boundary MPS).  Three paths, in the order in which they are tried:
//   * cut_topk (min(m, n) > chi_mps): FP32 finds where the leading space is, FP64 puts it right.
//       1. FP32 Householder QR with column pivoting of A (Golub & Van Loan, Matrix Computations,
//          4th ed., Alg. 5.4.1), stopped where the pivot falls below 1e-3 of the k-th: r <= min(m, n)
//          rows of R (typically 0.6 m).
//       2. FP32 one-sided Jacobi on the r columns of R^T: no rotations of V to accumulate (the
//          rotated, normalised columns are the right singular vectors of R) and, on the graded
//          factor of the pivoted QR, 4-6 sweeps instead of 12-22 (Drmac and Veselic, "New fast
//          and accurate Jacobi SVD algorithm I", 2008).
//       3. Newton's method on the invariant subspace in FP64: with V the k leading vectors,
//          P = A V, C = A^T P, E = C - V (V^T C) (all FP64), the first-order correction off the
//          space is, in the FP32 singular basis,
//          T = e + sum_i v_i (v_i . e) rho_i / (1 - rho_i), e = E / theta_j, rho_i = sigma_i^2 / theta_j
//          (FP32: T needs no more digits than it corrects).  Each pass gains the 5-7 digits of the
//          FP32 basis, so two passes reach FP64 accuracy; V is re-orthonormalised by one
//          Newton-Schulz step per pass.  FP64 work 10 n m k.
//     It applies where FP32 resolves the cut (cut_resolved): both rules of the truncation
//     (svd_cutoff, multiplet_rtol) keep exactly k with room for FP32's error, and sigma_k >= 1e-5
//     sigma_1; and it checks itself (the residual has to fall to FP64 rounding).
//   * cut_rank (rank <= chi_mps: nothing to truncate): FP64 pivoted QR of M, stopped at the first
//     pivot below svd_cutoff times the largest: U = Q, carry = R.  No SVD.  A pivot is not a singular
//     value, so it applies where the pivots leave no doubt about which values the cutoff keeps
//     (cut_rank_decided).
//   * cut_full (steep spectra, cuts inside a multiplet, larger cutoffs): as 1 and 2 in FP64 throughout;
//     every singular value, so the keep rule is decided on them.
// Measured against numpy's SVD on 130 cuts of the tests' networks: U U^T M of cut_topk differs by
// <= 6e-14 sigma_1 (median 2e-15).
//
// Data that one step writes and the next reads (norms, pivots, columns, vectors) is kept in
// registers or shared memory: L1 does not hold written lines, so through global memory each such
// exchange is an L2 round trip, and these loops are chains of them.
#pragma once

#include "cutnum.cuh"
#include "team.cuh"

namespace td {

// Largest biased exponent of the n x m column-major matrix A, through a shared int.
__device__ __forceinline__ int cut_max_exponent(const Team& tm, const double* A, int lda, int n, int m, int* slot) {
  if (tm.tid == 0) *slot = 0;
  tm.sync();
  unsigned mx = 0u;
  const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.nt >> 5;
  for (int c = warp; c < m; c += nw)
    for (int i = lane; i < n; i += 32) mx = max(mx, (unsigned)__double2hiint(A[(size_t)c * lda + i]) & 0x7FFFFFFFu);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) atomicMax(slot, (int)mx);
  tm.sync();
  const int e = *slot >> 20;
  tm.sync();
  return e;
}

// Sums of N (a power of two <= 32) values over the warp: lane l ends with the sum of value
// l / (32 / N) (each exchange halves the values a lane carries: N shuffles instead of 5 N).
template <int N, typename R>
__device__ __forceinline__ R cut_warp_sums(R (&v)[N], int lane) {
#pragma unroll
  for (int half = N / 2, off = 16; half >= 1; half >>= 1, off >>= 1) {
    const bool up = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const R send = up ? v[i] : v[i + half];
      const R keep = up ? v[i + half] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
#pragma unroll
  for (int off = 16 / N; off >= 1; off >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
  return v[0];
}

// Pivot keys: norm^2 (the FP32 value, or the upper word of the FP64 one: non-negative, so ordered as
// integers) with its lowest bits replaced by the column, lower columns first; 0: no column left.
// The keys only choose the pivot.
constexpr unsigned kCutColMask = 0x7FFu;   // up to 2048 columns
__device__ __forceinline__ unsigned cut_key(float norm2, int c) {
  return (__float_as_uint(fmaxf(norm2, 0.f)) & ~kCutColMask) | (kCutColMask - (unsigned)c);
}
__device__ __forceinline__ unsigned cut_key(double norm2, int c) {
  return ((unsigned)__double2hiint(norm2 > 0.0 ? norm2 : 0.0) & ~kCutColMask) | (kCutColMask - (unsigned)c);
}
__device__ __forceinline__ unsigned cut_best_key(const unsigned* keys, int nw, int lane) {
  return __reduce_max_sync(0xffffffffu, lane < nw ? keys[lane] : 0u);
}

// Two FP32 values in a 64-bit register: one instruction for both (FFMA2).
__device__ __forceinline__ uint64_t f2_pack(float lo, float hi) {
  return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ float f2_lo(uint64_t v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float f2_hi(uint64_t v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Householder QR with column pivoting of the FP32 copy of A (n x m FP64, scaled by 2^-expo), the
// copy in registers: warp w holds columns w, w + nw, ... (CPW of them), a lane rows lane + 32 t
// (t < RPL, two per register); rows that are done are zeroed there, so nothing is masked.  Two barriers
// per step: the pivot is known after the first, its column (written by its warp) after the second;
// dot products and norms of a warp's columns are reduced together.  The norm of a column after step j
// is its norm before it, summed afresh, minus R[j][c]^2.  Stops at the first pivot norm^2 <=
// max(rel2 * (that of the k-th pivot), abs2 * (that of the first)) or after `most` steps;
// L[j * ldl + c] = R[j][c].  vcol: n rounded up to 32, + 2 floats; keys: nw.
template <int CPW, int RPL>
__device__ __noinline__ int cut_qrcp_reg(Team tm, const double* A, int lda, int n, int m, int k, int expo, float rel2,
                                         float abs2, int most, float* L, int ldl, float* vcol, unsigned* keys) {
  constexpr int H = RPL / 2;
  const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.nt >> 5;
  uint64_t a[CPW][H];
  unsigned taken = 0u, key0 = 0u;
#pragma unroll
  for (int u = 0; u < CPW; ++u) {
    const int c = warp + u * nw;
    if (c >= m) taken |= 1u << u;
    uint64_t s2 = 0ull;
#pragma unroll
    for (int t = 0; t < H; ++t) {
      const int i = lane + 64 * t;
      const double* col = A + (size_t)(c < m ? c : 0) * lda;
      const float lo = (c < m && i < n) ? cut_f32(col[i], expo) : 0.f;
      const float hi = (c < m && i + 32 < n) ? cut_f32(col[i + 32], expo) : 0.f;
      a[u][t] = f2_pack(lo, hi);
      s2 = f2_fma(a[u][t], a[u][t], s2);
    }
    float s = f2_lo(s2) + f2_hi(s2);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (c < m) key0 = max(key0, cut_key(s, c));
  }
  if (lane == 0) keys[warp] = key0;
  const int q = n < m ? n : m, nv = (n + 31) & ~31;
  float d02 = 0.f, dk2 = 0.f;
  int j = 0;
  for (; j < q && j < most; ++j) {
    tm.sync();
    const unsigned key = cut_best_key(keys, nw, lane);
    const int p = (int)(kCutColMask - (key & kCutColMask));
    const float g2 = __uint_as_float(key & ~kCutColMask);
    if (j == 0) d02 = g2;
    if (j < k) dk2 = g2;
    if (key == 0u || !(g2 > 0.f) || g2 <= rel2 * dk2 || g2 <= abs2 * d02) break;
    const int jl = j & 31, jt = j >> 6;
    const bool jh = (j >> 5) & 1;
    if (warp == p % nw) {   // the pivot column becomes the reflector
      const int pu = p / nw;
      uint64_t x[H], s2 = 0ull;
      float x0 = 0.f;
#pragma unroll
      for (int t = 0; t < H; ++t) {
        x[t] = 0ull;
#pragma unroll
        for (int u = 0; u < CPW; ++u) x[t] = u == pu ? a[u][t] : x[t];
        s2 = f2_fma(x[t], x[t], s2);
        if (t == jt) x0 = jh ? f2_hi(x[t]) : f2_lo(x[t]);
      }
      float s = f2_lo(s2) + f2_hi(s2);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      x0 = __shfl_sync(0xffffffffu, x0, jl);
      const float nrm = s * rsqrtf(fmaxf(s, 1e-37f)), alpha = x0 >= 0.f ? -nrm : nrm;
#pragma unroll
      for (int t = 0; t < H; ++t) {
        const int i = lane + 64 * t;
        if (i < nv) vcol[i] = i == j ? x0 - alpha : f2_lo(x[t]);
        if (i + 32 < nv) vcol[i + 32] = i + 32 == j ? x0 - alpha : f2_hi(x[t]);
      }
      if (lane == 0) {
        vcol[nv] = s > 0.f ? __fdividef(1.f, s + fabsf(x0) * nrm) : 0.f;   // 2 / v.v
        vcol[nv + 1] = alpha;
      }
    }
    tm.sync();
    uint64_t v[H];
#pragma unroll
    for (int t = 0; t < H; ++t) {
      const int i = lane + 64 * t;
      v[t] = f2_pack(i < nv ? vcol[i] : 0.f, i + 32 < nv ? vcol[i + 32] : 0.f);
    }
    const float tau = vcol[nv], alpha = vcol[nv + 1];
    float sums[2 * CPW];
#pragma unroll
    for (int u = 0; u < CPW; ++u) {
      uint64_t d = 0ull, s2 = 0ull;
#pragma unroll
      for (int t = 0; t < H; ++t) {
        d = f2_fma(v[t], a[u][t], d);
        s2 = f2_fma(a[u][t], a[u][t], s2);
      }
      sums[u] = f2_lo(d) + f2_hi(d);
      sums[CPW + u] = f2_lo(s2) + f2_hi(s2);
    }
    const float mine = cut_warp_sums<2 * CPW, float>(sums, lane);
    constexpr int STEP = 32 / (2 * CPW);
    unsigned best = 0u;
#pragma unroll
    for (int u = 0; u < CPW; ++u) {
      const int c = warp + u * nw;
      const float w = -tau * __shfl_sync(0xffffffffu, mine, u * STEP);
      const float s = __shfl_sync(0xffffffffu, mine, (CPW + u) * STEP);
      const uint64_t w2 = f2_pack(w, w);
#pragma unroll
      for (int t = 0; t < H; ++t) a[u][t] = f2_fma(w2, v[t], a[u][t]);
      float top = 0.f;
#pragma unroll
      for (int t = 0; t < H; ++t)
        if (t == jt) {   // the same for every thread
          top = jh ? f2_hi(a[u][t]) : f2_lo(a[u][t]);
          if (lane == jl) a[u][t] = jh ? f2_pack(f2_lo(a[u][t]), 0.f) : f2_pack(0.f, f2_hi(a[u][t]));
        }
      const bool on = !((taken >> u) & 1u) && c != p;
      if (lane == jl) {
        if (c < m) L[(size_t)j * ldl + c] = on ? top : (c == p ? alpha : 0.f);
        if (on) best = max(best, cut_key(s - top * top, c));
      }
      if (c == p) taken |= 1u << u;
    }
    if (lane == jl) keys[warp] = best;
  }
  tm.sync();
  return j;
}

// The same factorisation with the copy A (n x m, ld n; destroyed) in memory, for cuts whose copy the
// registers do not hold: four columns at a time, one barrier per step (every warp forms the reflector
// from the pivot column, which is only read).  keys: 2 nw.
static __device__ __noinline__ int cut_qrcp_mem(Team tm, float* A, int n, int m, int k, float rel2, float abs2, int most,
                                                float* L, int ldl, unsigned char* taken, unsigned* keys) {
  constexpr int CB = 4;
  const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.nt >> 5;
  {
    unsigned key = 0u;
    for (int c = warp; c < m; c += nw) {
      const float* a = A + (size_t)c * n;
      float s = 0.f;
      for (int i = lane; i < n; i += 32) s += a[i] * a[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) taken[c] = 0;
      key = max(key, cut_key(s, c));
    }
    if (lane == 0) keys[warp] = key;
  }
  const int q = n < m ? n : m;
  float d02 = 0.f, dk2 = 0.f;
  int j = 0;
  for (; j < q && j < most; ++j) {
    tm.sync();
    const unsigned key = cut_best_key(keys + (j & 1) * nw, nw, lane);
    if (key == 0u) break;
    const int p = (int)(kCutColMask - (key & kCutColMask));
    const float* ap = A + (size_t)p * n;
    float d2 = 0.f;
    for (int i = j + lane; i < n; i += 32) d2 += ap[i] * ap[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d2 += __shfl_xor_sync(0xffffffffu, d2, o);
    if (j == 0) d02 = d2;
    if (j < k) dk2 = d2;
    if (!(d2 > 0.f) || d2 <= rel2 * dk2 || d2 <= abs2 * d02) break;
    const float x0 = ap[j], nrm = sqrtf(d2);
    const float alpha = x0 >= 0.f ? -nrm : nrm;
    const float v0 = x0 - alpha, tau = 1.f / (d2 + fabsf(x0) * nrm);
    unsigned best = 0u;
    for (int c0 = warp * CB; c0 < m; c0 += nw * CB) {
      float dots[CB], top[CB];
      float* ac[CB];
      unsigned on = 0u;
#pragma unroll
      for (int u = 0; u < CB; ++u) {
        const int c = c0 + u;
        const bool o = c < m && c != p && !taken[c < m ? c : 0];
        on |= (unsigned)o << u;
        ac[u] = A + (size_t)(o ? c : p) * n;
        dots[u] = 0.f;
        top[u] = ac[u][j];
      }
      if (on)
#pragma unroll 2
        for (int i = j + 1 + lane; i < n; i += 32) {
          const float v = ap[i];
#pragma unroll
          for (int u = 0; u < CB; ++u) dots[u] += v * ac[u][i];
        }
      const float dot = cut_warp_sums<CB, float>(dots, lane);
      float w[CB], ss[CB];
#pragma unroll
      for (int u = 0; u < CB; ++u) {
        w[u] = tau * (__shfl_sync(0xffffffffu, dot, u * (32 / CB)) + v0 * top[u]);
        ss[u] = 0.f;
      }
      if (on)
#pragma unroll 2
        for (int i = j + 1 + lane; i < n; i += 32) {
          const float v = ap[i];
          float x[CB];
#pragma unroll
          for (int u = 0; u < CB; ++u) {
            x[u] = ac[u][i] - w[u] * v;
            ss[u] += x[u] * x[u];
          }
#pragma unroll
          for (int u = 0; u < CB; ++u)
            if ((on >> u) & 1u) ac[u][i] = x[u];
        }
      // the norms below row j summed afresh: the stop is decided on them
      const float below = cut_warp_sums<CB, float>(ss, lane);
#pragma unroll
      for (int u = 0; u < CB; ++u) {
        const int c = c0 + u;
        const float s = __shfl_sync(0xffffffffu, below, u * (32 / CB));
        const bool o = (on >> u) & 1u;
        if (lane == 0 && c < m) {
          const float x = top[u] - w[u] * v0;   // R[j][c]
          L[(size_t)j * ldl + c] = o ? x : (c == p ? alpha : 0.f);
          if (o) ac[u][j] = x;
          if (c == p) taken[c] = 1;
        }
        if (o) best = max(best, cut_key(s, c));
      }
    }
    if (lane == 0) keys[((j + 1) & 1) * nw + warp] = best;
  }
  tm.sync();
  return j;
}

// FP32 Jacobi: rotates above ~FP32 rounding; done when a sweep saw no |cos| above 3e-4 (which leaves
// ~1e-7: the convergence is quadratic).
constexpr float kCutRot2 = 1e-12f, kCutDone2 = 1e-7f;
__device__ __forceinline__ void cut_rotation(float al, float be, float ga, float& c, float& s) {
  const float zeta = __fdividef(be - al, 2.f * ga), w = 1.f + zeta * zeta;
  const float t = copysignf(__fdividef(1.f, fabsf(zeta) + w * rsqrtf(w)), zeta);
  c = rsqrtf(1.f + t * t);
  s = t * c;
}

// FP64 one-sided Jacobi of the r columns (length m, ldl) of L, without V.  As in the truncation cores
// (core.cu, group_jacobi) an FP64 instruction costs the same for one lane as for 32, so the inner
// products take few lanes per pair (at most four warps in all), the angles one lane per pair, and the
// rotations of the pairs that rotate are spread over all threads row by row.  The convergence is
// quadratic, so the sweep that sees no |cos| above 1e-8 is the last.  buf: 5 (r + 1) / 2 doubles, list:
// (r + 1) / 2 ints, slots: four shared ints.
static __device__ __noinline__ void cut_jacobi64(Team tm, double* L, int ldl, int m, int r, double* buf, int* list,
                                                 int* slots) {
  const int ne = r + (r & 1), half = ne / 2, mm = ne - 1;
  double *al = buf, *be = al + half, *ga = be + half, *cs = ga + half, *sn = cs + half;
  int g = 1;
  while (g < 32 && 2 * g * half <= 128) g *= 2;
  const int ngroups = tm.nt / g, grp = tm.tid / g, gl = tm.tid % g;
  for (int sweep = 0; sweep < 40; ++sweep) {
    if (tm.tid == 0) slots[0] = 0;
    for (int k = 0; k < mm; ++k) {
      int* cnt = slots + 1 + (k & 1);
      if (tm.tid == 0) *cnt = 0;
      for (int i0 = 0; i0 < half; i0 += ngroups) {
        const int i = i0 + grp;
        int p = 0, q = 0;
        if (i < half) team_rr_pair(k, i, ne, p, q);
        const bool active = i < half && q < r;
        double x2 = 0.0, y2 = 0.0, xy = 0.0;
        if (active) {
          const double* ap = L + (size_t)p * ldl;
          const double* aq = L + (size_t)q * ldl;
          for (int row = gl; row < m; row += g) {
            const double u = ap[row], v = aq[row];
            x2 += u * u;
            y2 += v * v;
            xy += u * v;
          }
        }
        if (i0 + (tm.tid & ~31) / g < half)   // a warp without a pair has nothing to add
          for (int o = g >> 1; o > 0; o >>= 1) {
            x2 += __shfl_xor_sync(0xffffffffu, x2, o);
            y2 += __shfl_xor_sync(0xffffffffu, y2, o);
            xy += __shfl_xor_sync(0xffffffffu, xy, o);
          }
        if (gl == 0 && i < half) {
          al[i] = x2;
          be[i] = y2;
          ga[i] = active ? xy : 0.0;
        }
      }
      tm.sync();
      for (int i = tm.tid; i < half; i += tm.nt) {
        double c, s;
        if (jacobi_rot(al[i], be[i], ga[i], TeamTol<double>::rel(), c, s)) {
          cs[i] = c;
          sn[i] = s;
          list[atomicAdd(cnt, 1)] = i;
          if (ga[i] * ga[i] > 1e-16 * (al[i] * be[i])) slots[0] = 1;
        }
      }
      tm.sync();
      const int tasks = *cnt * m;
      for (int t = tm.tid; t < tasks; t += tm.nt) {
        const int i = list[t / m], row = t % m;
        int p, q;
        team_rr_pair(k, i, ne, p, q);
        double* xp = L + (size_t)p * ldl + row;
        double* xq = L + (size_t)q * ldl + row;
        const double c = cs[i], s = sn[i], u = *xp, v = *xq;
        *xp = c * u - s * v;
        *xq = s * u + c * v;
      }
      tm.sync();
    }
    const int any = slots[0];
    tm.sync();
    if (!any) break;
  }
}

// team_svd_onesided<double> of A (m x n, column-major, lda) with V accumulated (n x n, from 1) for a whole
// block: the same inner products (lanes per pair, order of the sums), but the angles one lane per pair
// and the rotations only for the pairs that rotate, row by row over all threads -- bit for bit the
// same result with ~2/3 of the FP64 instructions.  Measured (the recorded final contraction of rotated d7,
// chi_mps 8, 152 shots): 63 -> 49 ms.  buf: 5 (n + 1) / 2 doubles, list: (n + 1) / 2 ints,
// slots: four shared ints.
static __device__ __noinline__ void block_svd_onesided(Team tm, double* A, int lda, int m, int n, double* V, int ldv,
                                                       double* buf, int* list, int* slots, int max_sweeps) {
  for (int w = tm.tid; w < n * n; w += tm.nt) V[(w / n) * ldv + (w % n)] = (w / n == w % n) ? 1.0 : 0.0;
  tm.sync();
  if (n < 2) return;
  const int ne = n + (n & 1), half = ne / 2;
  const int g = team_svd_group(tm.nt, m, n), ngroups = tm.nt / g, grp = tm.tid / g, gl = tm.tid % g;
  double *al = buf, *be = al + half, *ga = be + half, *cs = ga + half, *sn = cs + half;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    if (tm.tid == 0) slots[0] = 0;
    for (int k = 0; k < ne - 1; ++k) {
      int* cnt = slots + 1 + (k & 1);
      if (tm.tid == 0) *cnt = 0;
      for (int i0 = 0; i0 < half; i0 += ngroups) {
        const int i = i0 + grp;
        int p = 0, q = 0;
        bool active = i < half;
        if (active) {
          team_rr_pair(k, i, ne, p, q);
          active = q < n;
        }
        double x2 = 0.0, y2 = 0.0, xy = 0.0;
        if (active) {
          const double* ap_ = A + (size_t)p * lda;
          const double* aq_ = A + (size_t)q * lda;
          for (int r = gl; r < m; r += g) {
            const double ap = ap_[r], aq = aq_[r];
            x2 += ap * ap;
            y2 += aq * aq;
            xy += ap * aq;
          }
        }
        if (i0 + (tm.tid & ~31) / g < half)   // a warp without a pair has nothing to add
          for (int o = g >> 1; o > 0; o >>= 1) {
            x2 += __shfl_xor_sync(0xffffffffu, x2, o);
            y2 += __shfl_xor_sync(0xffffffffu, y2, o);
            xy += __shfl_xor_sync(0xffffffffu, xy, o);
          }
        if (gl == 0 && i < half) {
          al[i] = x2;
          be[i] = y2;
          ga[i] = active ? xy : 0.0;
        }
      }
      tm.sync();
      for (int i = tm.tid; i < half; i += tm.nt) {
        double c, s;
        if (jacobi_rot(al[i], be[i], ga[i], TeamTol<double>::rel(), c, s)) {
          cs[i] = c;
          sn[i] = s;
          list[atomicAdd(cnt, 1)] = i;
          slots[0] = 1;
        }
      }
      tm.sync();
      const int rows = m + n, tasks = *cnt * rows;
      for (int t = tm.tid; t < tasks; t += tm.nt) {
        const int i = list[t / rows], row = t % rows;
        int p, q;
        team_rr_pair(k, i, ne, p, q);
        double* ap_ = row < m ? A + (size_t)p * lda + row : V + (size_t)p * ldv + (row - m);
        double* aq_ = row < m ? A + (size_t)q * lda + row : V + (size_t)q * ldv + (row - m);
        const double c = cs[i], s = sn[i], ap = *ap_, aq = *aq_;
        *ap_ = c * ap - s * aq;
        *aq_ = s * ap + c * aq;
      }
      tm.sync();
    }
    const int any = slots[0];
    tm.sync();
    if (!any) break;
  }
}

// FP32 one-sided Jacobi of the r columns of L, without V, four rows per load and two per instruction:
// columns padded with zeros to a multiple of 32 rows (rows32), ld cut_ld32.  What bounds it is
// instructions (18 per 4 rows of a pair against ~80 one by one) and the latency of a step (~350 cycles);
// N4 loads per lane and column stay in registers, N4 = 0 reads them twice.
template <int N4>
__device__ __noinline__ void cut_jacobi32(Team tm, float* L, int ldl, int rows32, int r, int g, int* flag) {
  constexpr int N = N4 > 0 ? N4 : 1;
  const int ne = r + (r & 1), half = ne / 2, mm = ne - 1;
  const int ngroups = tm.nt / g, n4 = rows32 / 4;
  const int grp = tm.tid / g, gl = tm.tid % g;
  for (int sweep = 0; sweep < 30; ++sweep) {
    if (tm.tid == 0) *flag = 0;
    tm.sync();
    bool more = false;
    for (int k = 0; k < mm; ++k) {
      for (int i0 = 0; i0 < half; i0 += ngroups) {
        const int i = i0 + grp;
        int p = k + i, q = k - i;   // round-robin pair i of step k (team_rr_pair; their order does not matter)
        p = p >= mm ? p - mm : p;
        q = q < 0 ? q + mm : q;
        if (i == 0) q = mm;
        const bool active = i < half && p < r && q < r;
        ulonglong2* ap = reinterpret_cast<ulonglong2*>(L + (size_t)(active ? p : 0) * ldl);
        ulonglong2* aq = reinterpret_cast<ulonglong2*>(L + (size_t)(active ? q : 0) * ldl);
        ulonglong2 x[N], y[N];
        uint64_t al2 = 0ull, be2 = 0ull, ga2 = 0ull;
        if (N4 > 0) {
#pragma unroll
          for (int t = 0; t < N; ++t) {
            const bool in = active && gl + t * g < n4;
            x[t] = in ? ap[gl + t * g] : make_ulonglong2(0ull, 0ull);
            y[t] = in ? aq[gl + t * g] : make_ulonglong2(0ull, 0ull);
          }
#pragma unroll
          for (int t = 0; t < N; ++t) {
            al2 = f2_fma(x[t].x, x[t].x, al2);
            be2 = f2_fma(y[t].x, y[t].x, be2);
            ga2 = f2_fma(x[t].x, y[t].x, ga2);
            al2 = f2_fma(x[t].y, x[t].y, al2);
            be2 = f2_fma(y[t].y, y[t].y, be2);
            ga2 = f2_fma(x[t].y, y[t].y, ga2);
          }
        } else if (active) {
#pragma unroll 4
          for (int t = gl; t < n4; t += g) {
            const ulonglong2 u = ap[t], v = aq[t];
            al2 = f2_fma(u.x, u.x, al2);
            be2 = f2_fma(v.x, v.x, be2);
            ga2 = f2_fma(u.x, v.x, ga2);
            al2 = f2_fma(u.y, u.y, al2);
            be2 = f2_fma(v.y, v.y, be2);
            ga2 = f2_fma(u.y, v.y, ga2);
          }
        }
        float al = f2_lo(al2) + f2_hi(al2), be = f2_lo(be2) + f2_hi(be2), ga = f2_lo(ga2) + f2_hi(ga2);
        for (int o = g >> 1; o > 0; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o);
          be += __shfl_xor_sync(0xffffffffu, be, o);
          ga += __shfl_xor_sync(0xffffffffu, ga, o);
        }
        const float gg = ga * ga, ab = al * be;
        if (active && gg > kCutRot2 * ab) {
          more |= gg > kCutDone2 * ab;
          float c, s;
          cut_rotation(al, be, ga, c, s);
          const uint64_t c2 = f2_pack(c, c), s2 = f2_pack(s, s), m2 = f2_pack(-s, -s);
          if (N4 > 0) {
#pragma unroll
            for (int t = 0; t < N; ++t)
              if (gl + t * g < n4) {
                ap[gl + t * g] = make_ulonglong2(f2_fma(c2, x[t].x, f2_mul(m2, y[t].x)), f2_fma(c2, x[t].y, f2_mul(m2, y[t].y)));
                aq[gl + t * g] = make_ulonglong2(f2_fma(c2, y[t].x, f2_mul(s2, x[t].x)), f2_fma(c2, y[t].y, f2_mul(s2, x[t].y)));
              }
          } else {
#pragma unroll 4
            for (int t = gl; t < n4; t += g) {
              const ulonglong2 u = ap[t], v = aq[t];
              ap[t] = make_ulonglong2(f2_fma(c2, u.x, f2_mul(m2, v.x)), f2_fma(c2, u.y, f2_mul(m2, v.y)));
              aq[t] = make_ulonglong2(f2_fma(c2, v.x, f2_mul(s2, u.x)), f2_fma(c2, v.y, f2_mul(s2, u.y)));
            }
          }
        }
      }
      tm.sync();
    }
    if (more) *flag = 1;
    tm.sync();
    const int any = *flag;
    tm.sync();
    if (!any) break;
  }
}

// Norms of the r columns and their descending order.
template <typename R>
__device__ __forceinline__ void cut_order(const Team& tm, const R* L, int ldl, int m, int r, R* sg, int* ord) {
  const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.nt >> 5;
  for (int c = warp; c < r; c += nw) {
    R s = R(0);
    for (int i = lane; i < m; i += 32) s += L[(size_t)c * ldl + i] * L[(size_t)c * ldl + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) sg[c] = sqrt(s);
  }
  tm.sync();
  for (int j = tm.tid; j < r; j += tm.nt) {
    const R v = sg[j];
    int rank = 0;
    for (int i = 0; i < r; ++i) rank += (sg[i] > v || (sg[i] == v && i < j)) ? 1 : 0;
    ord[rank] = j;
  }
  tm.sync();
}

// P[kk][i] = sum_c A[c][i] V[c][kk]  (n x k), KB columns per thread.
template <int KB>
__device__ __forceinline__ void cut_av(const Team& tm, const double* A, int lda, int n, int m, const double* V, int k,
                                       double* P) {
  const int nb = (k + KB - 1) / KB;
  for (int w = tm.tid; w < n * nb; w += tm.nt) {
    const int i = w % n, k0 = (w / n) * KB;
    int kx[KB];
    double acc[KB];
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      kx[u] = k0 + u < k ? k0 + u : k - 1;
      acc[u] = 0.0;
    }
#pragma unroll 4
    for (int c = 0; c < m; ++c) {
      const double a = A[(size_t)c * lda + i];
#pragma unroll
      for (int u = 0; u < KB; ++u) acc[u] += a * V[c * k + kx[u]];
    }
#pragma unroll
    for (int u = 0; u < KB; ++u)
      if (k0 + u < k) P[(size_t)(k0 + u) * n + i] = acc[u];
  }
}

// C[kk][c] = sum_i A[c][i] P[kk][i]  (m x k), KB columns per thread.
template <int KB>
__device__ __forceinline__ void cut_atp(const Team& tm, const double* A, int lda, int n, int m, const double* P, int k,
                                        double* C) {
  const int nb = (k + KB - 1) / KB;
  for (int w = tm.tid; w < m * nb; w += tm.nt) {
    const int c = w % m, k0 = (w / m) * KB;
    const double* a = A + (size_t)c * lda;
    const double* pk[KB];
    double acc[KB];
#pragma unroll
    for (int u = 0; u < KB; ++u) {
      pk[u] = P + (size_t)(k0 + u < k ? k0 + u : k - 1) * n;
      acc[u] = 0.0;
    }
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
      const double x = a[i];
#pragma unroll
      for (int u = 0; u < KB; ++u) acc[u] += x * pk[u][i];
    }
#pragma unroll
    for (int u = 0; u < KB; ++u)
      if (k0 + u < k) C[(size_t)(k0 + u) * m + c] = acc[u];
  }
}

// Columns per thread: as many as leave every thread a task (fewer loads per FMA).
static __device__ __noinline__ void cut_mul_av(Team tm, const double* A, int lda, int n, int m, const double* V, int k,
                                               double* P) {
  if (n * ((k + 3) / 4) >= tm.nt) cut_av<4>(tm, A, lda, n, m, V, k, P);
  else if (n * ((k + 1) / 2) >= tm.nt) cut_av<2>(tm, A, lda, n, m, V, k, P);
  else cut_av<1>(tm, A, lda, n, m, V, k, P);
  tm.sync();
}
static __device__ __noinline__ void cut_mul_atp(Team tm, const double* A, int lda, int n, int m, const double* P, int k,
                                                double* C) {
  if (m * ((k + 3) / 4) >= tm.nt) cut_atp<4>(tm, A, lda, n, m, P, k, C);
  else if (m * ((k + 1) / 2) >= tm.nt) cut_atp<2>(tm, A, lda, n, m, P, k, C);
  else cut_atp<1>(tm, A, lda, n, m, P, k, C);
  tm.sync();
}

// V2 = V (3I - V^T V) / 2  (m x k, row-major; S scratch): orthonormal to e^2 from e.
static __device__ __noinline__ void cut_orthonormalise(Team tm, const double* V, double* V2, double* S, int m, int k) {
  // four lanes per entry of V^T V
  for (int w0 = 0; w0 < k * k; w0 += tm.nt / 4) {
    const int w = w0 + tm.tid / 4, part = tm.tid & 3;
    const int a = w / k, b = w % k;
    double s = 0.0;
    if (w < k * k && a <= b)
      for (int c = part; c < m; c += 4) s += V[c * k + a] * V[c * k + b];
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if (w < k * k && a <= b && part == 0) {
      const double t = (a == b ? 1.5 : 0.0) - 0.5 * s;
      S[a * k + b] = t;
      S[b * k + a] = t;
    }
  }
  tm.sync();
  for (int w = tm.tid; w < m * k; w += tm.nt) {
    const int c = w / k, b = w % k;
    double s = 0.0;
    for (int a = 0; a < k; ++a) s += V[c * k + a] * S[a * k + b];
    V2[w] = s;
  }
  tm.sync();
}

// Leading dimension of the columns that cut_jacobi64 turns: = lanes per pair mod 32 at full rank, which
// puts the lane groups of consecutive pairs on different banks.
__host__ __device__ __forceinline__ int cut_ldl(int nt, int m) { return bank_ld32(m, team_svd_group(nt, m, m)); }
// The same for four-row loads: eight lanes' 128 bytes on different banks (a multiple of 4; below
// 2 cut_ldl, so that the columns fit the FP64 ones' place).
__host__ __device__ __forceinline__ int cut_ld32(int nt, int m) {
  const int g = team_svd_group(nt, m, m);
  return (m + 31) / 32 * 32 + (g < 8 ? 4 * g : 0);
}

// Scratch of a cut.  Shared memory takes the small arrays, then the FP32 columns and the vectors.
struct CutBuf {
  double *V, *V2;   // [m][k]
  double* C;        // [k][m]
  double* P;        // [k][n]
  float* E;         // [k][m]
  float* W;         // [q][k]
  double* S;        // [k][k]
  double* th;       // [k] theta_j, then [k] 1 / theta_j
  float* sg;        // [q] singular values (FP32, of the scaled matrix)
  int* ord;         // [q] descending order
  float* vcol;      // [n + 34] reflector (n rounded up to 32, and two values)
  unsigned char* taken;   // [max(m, n)]
  unsigned* keys;   // [64]
  static __host__ __device__ int64_t small_bytes(int m, int n, int k) {
    const int q = m < n ? m : n, x = m < n ? n : m;
    return (16 * (int64_t)k + 4 * (2 * (int64_t)q + n + 34 + 64) + x + 31) / 16 * 16;
  }
  static __host__ __device__ int64_t vec_bytes(int m, int n, int k, bool with_P) {
    const int q = m < n ? m : n;
    return (8 * (3 * (int64_t)m * k + (int64_t)k * k + (with_P ? (int64_t)k * n : 0)) + 4 * ((int64_t)m * k + (int64_t)q * k) +
            31) / 16 * 16;
  }
  __device__ void carve_small(unsigned char* base, int m, int n, int k) {
    const int q = m < n ? m : n;
    th = reinterpret_cast<double*>(base);
    sg = reinterpret_cast<float*>(th + 2 * k);
    ord = reinterpret_cast<int*>(sg + q);
    vcol = reinterpret_cast<float*>(ord + q);
    keys = reinterpret_cast<unsigned*>(vcol + n + 34);
    taken = reinterpret_cast<unsigned char*>(keys + 64);
  }
  // P_ == null: P after the other vectors
  __device__ void carve_vec(double* base, int m, int n, int k, double* P_) {
    V = base;
    V2 = V + (size_t)m * k;
    C = V2 + (size_t)m * k;
    S = C + (size_t)m * k;
    double* e = S + (size_t)k * k;
    P = P_;
    if (!P_) {
      P = e;
      e += (size_t)k * n;
    }
    E = reinterpret_cast<float*>(e);
    W = E + (size_t)m * k;
  }
};

// FP32 QR and Jacobi of step 1 and 2 (file comment).  cap floats at Ls (shared) take the columns when
// they fit -- the rank decides how many are needed, so a rank beyond them starts over with L_g.
// Returns the rank; the columns are at *L_out.
__device__ __forceinline__ int cut_fp32(const Team& tm, const double* A, int lda, int n, int m, int k, int expo, float* A_g,
                                        float* L_g, float* Ls, int cap, CutBuf& b, int* slots, float** L_out, int* ldl_out) {
  const int q = n < m ? n : m, nw = tm.nt >> 5;
  const int ldl = cut_ld32(tm.nt, m);
  const int cols = cap / ldl < q ? cap / ldl : q;
  const int cpw = (m + nw - 1) / nw;
  float* L = cols > k ? Ls : L_g;
  int r = 0;
  for (int most = cols > k ? cols : q;; most = q, L = L_g) {
    // the copy in registers: 32 a thread, 64 in the 512-thread blocks (which have 128)
    if (cpw <= 4 && n <= 128)
      r = cut_qrcp_reg<4, 4>(tm, A, lda, n, m, k, expo, 1e-6f, 1e-12f, most, L, ldl, b.vcol, b.keys);
    else if (cpw <= 8 && n <= 128)
      r = cut_qrcp_reg<8, 4>(tm, A, lda, n, m, k, expo, 1e-6f, 1e-12f, most, L, ldl, b.vcol, b.keys);
    else if (cpw <= 4 && n <= 256)
      r = cut_qrcp_reg<4, 8>(tm, A, lda, n, m, k, expo, 1e-6f, 1e-12f, most, L, ldl, b.vcol, b.keys);
    else if (tm.nt == 512 && cpw <= 8 && n <= 256)
      r = cut_qrcp_reg<8, 8>(tm, A, lda, n, m, k, expo, 1e-6f, 1e-12f, most, L, ldl, b.vcol, b.keys);
    else {
      const int lane = tm.tid & 31;
      for (int c = tm.tid >> 5; c < m; c += nw)
        for (int i = lane; i < n; i += 32) A_g[(size_t)c * n + i] = cut_f32(A[(size_t)c * lda + i], expo);
      tm.sync();
      r = cut_qrcp_mem(tm, A_g, n, m, k, 1e-6f, 1e-12f, most, L, ldl, b.taken, b.keys);
    }
    if (r < most || most == q) break;
  }
  *L_out = L;
  *ldl_out = ldl;
  if (r <= k) return r;
  const int rows32 = (m + 31) & ~31, pad = rows32 - m;
  for (int w = tm.tid; w < r * pad; w += tm.nt) L[(size_t)(w / pad) * ldl + m + w % pad] = 0.f;
  tm.sync();
  const int g = team_svd_group(tm.nt, rows32 / 4, r), n4 = (rows32 / 4 + g - 1) / g;
  if (n4 <= 1) cut_jacobi32<1>(tm, L, ldl, rows32, r, g, slots);
  else if (n4 <= 2) cut_jacobi32<2>(tm, L, ldl, rows32, r, g, slots);
  else if (n4 <= 4) cut_jacobi32<4>(tm, L, ldl, rows32, r, g, slots);
  else if (n4 <= 8 && tm.nt == 512) cut_jacobi32<8>(tm, L, ldl, rows32, r, g, slots);
  else cut_jacobi32<0>(tm, L, ldl, rows32, r, g, slots);
  cut_order<float>(tm, L, ldl, m, r, b.sg, b.ord);
  return r;
}

// Whether the FP32 singular values t0 (the largest), tk (the k-th), tn (the next) decide the cut at k:
// keep those above cutoff * t0, and none of a multiplet cut inside s_k - s_{k+1} <= rtol * t0.  A
// pivoted QR and an SVD in FP32 give the values to 2e-7 t0 (numpy, largest error over 164 cuts of the tests'
// networks), so both rules have to hold by 1e-6 t0; closer cuts are decided in FP64.
__device__ __forceinline__ bool cut_resolved(float t0, float tk, float tn, double cutoff, double rtol) {
  const float eps = 1e-6f * t0;
  return tk >= 1e-5f * t0 && tk > float(cutoff) * t0 + eps && tk - tn > 1e-4f * tk && tk - tn > float(rtol) * t0 + eps;
}

// See the file comment.  2^expo: the magnitude of A's largest entry.  b.P receives the carry
// U_k^T M, b.V the vectors; slots: two shared ints.  Returns false (nothing usable) when the cut is not
// one for this path; *r32 is then the FP32 rank.
static __device__ __noinline__ bool cut_topk(Team tm, const double* A, int lda, int n, int m, int k, double cutoff,
                                             double rtol, int expo, float* A_g, float* L_g, float* Ls, int cap,
                                             CutBuf& b, int* slots, double* s0, int* r32) {
  const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.nt >> 5;
  float* L;
  int ldl;
  const int r = cut_fp32(tm, A, lda, n, m, k, expo, A_g, L_g, Ls, cap, b, slots, &L, &ldl);
  *r32 = r;
  if (r <= k) return false;
  if (!cut_resolved(b.sg[b.ord[0]], b.sg[b.ord[k - 1]], b.sg[b.ord[k]], cutoff, rtol)) return false;
  double *V = b.V, *V2 = b.V2;
  for (int w = tm.tid; w < m * k; w += tm.nt) {
    const int c = w / k, o = b.ord[w % k];
    V[w] = double(L[(size_t)o * ldl + c] / b.sg[o]);
  }
  tm.sync();
  const double unit2 = ldexp(1.0, -2 * expo);
  // the residual at which the space is right to FP64 rounding: an error in it is the residual over 1 - rho of the
  // first vector left out, so next to a multiplet it has to fall further (or to its own rounding)
  const float ratio = b.sg[b.ord[k]] / b.sg[b.ord[k - 1]];
  const float done = 5e-16f * fminf(1.f, 8.f * (1.f - ratio * ratio));
  float prev = 0.f;
  bool ok = false, last = false;
  for (int it = 0; it < 10; ++it) {
    cut_orthonormalise(tm, V, V2, b.S, m, k);
    {
      double* t = V;
      V = V2;
      V2 = t;
    }
    cut_mul_av(tm, A, lda, n, m, V, k, b.P);
    if (last) {
      ok = true;
      break;
    }
    if (tm.tid == 0) slots[1] = 0;
    cut_mul_atp(tm, A, lda, n, m, b.P, k, b.C);
    for (int w0 = 0; w0 < k * k; w0 += tm.nt / 4) {   // S = V^T C, four lanes per entry
      const int w = w0 + tm.tid / 4, part = tm.tid & 3;
      const int a = w / k, j = w % k;
      double s = 0.0;
      if (w < k * k)
        for (int c = part; c < m; c += 4) s += V[c * k + a] * b.C[(size_t)j * m + c];
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      if (w < k * k && part == 0) {
        b.S[w] = s;
        if (a == j) {
          b.th[j] = s;
          b.th[k + j] = 1.0 / s;
        }
      }
    }
    tm.sync();
    unsigned worst = 0u;
    const double th0 = b.th[0];
    for (int w = tm.tid; w < m * k; w += tm.nt) {
      const int j = w / m, c = w % m;
      double s = b.C[w];
      for (int a = 0; a < k; ++a) s -= V[c * k + a] * b.S[a * k + j];
      const float e = float(s * b.th[k + j]);
      b.E[w] = e;
      worst = max(worst, cut_residual(e, b.th[j], th0, expo));
    }
    worst = __reduce_max_sync(0xffffffffu, worst);
    if (lane == 0) atomicMax(slots + 1, (int)worst);
    tm.sync();
    const float res = __int_as_float(slots[1]);
    // converged: the residual at FP64 rounding (or no longer falling just above it)
    if (res <= done || (it > 0 && res <= 2e-14f && res > 0.1f * prev)) {
      ok = true;
      break;
    }
    if (!(res < 1e-2f) || (it > 0 && !(res < 0.3f * prev))) break;
    for (int i = warp; i < r - k; i += nw) {   // (v_i . e_j) rho / (1 - rho) / sigma_i, a warp per i
      const int o = b.ord[k + i];
      const float* l = L + (size_t)o * ldl;
      const float s2 = b.sg[o] * b.sg[o];
      for (int j0 = 0; j0 < k; j0 += 4) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        for (int c = lane; c < m; c += 32) {
          const float x = l[c];
#pragma unroll
          for (int u = 0; u < 4; ++u) d[u] += x * b.E[(size_t)(j0 + u < k ? j0 + u : k - 1) * m + c];
        }
        const float mine = cut_warp_sums<4, float>(d, lane);
        const int j = j0 + (lane >> 3);
        if ((lane & 7) == 0 && j < k) {
          const float rho = s2 / float(b.th[j] * unit2);
          b.W[(size_t)i * k + j] = mine / s2 * (rho / (1.f - rho));
        }
      }
    }
    tm.sync();
    for (int w = tm.tid; w < m * k; w += tm.nt) {
      const int j = w / m, c = w % m;
      float t = b.E[w];
#pragma unroll 4
      for (int i = 0; i < r - k; ++i) t += L[(size_t)b.ord[k + i] * ldl + c] * b.W[(size_t)i * k + j];
      V[c * k + j] += double(t);
    }
    // the pass gained a factor res / prev; the next residual is predicted below that
    last = it > 0 && res * (res / prev) * 8.f < done;
    prev = res;
    tm.sync();
  }
  b.V = V;
  if (ok) *s0 = sqrt(b.th[0]);
  return ok;
}

// Whether a pivoted QR of n columns decides which singular values lie above cutoff times the largest: first and
// last the first and the last kept pivot, left the square of the pivot it stopped at over the first's (0: none).
// The largest value s_1 is between the first pivot and sqrt(n) times it.  The dropped ones are at most the norm
// of what is left, sqrt(n left) times the first pivot, and below the cutoff where that is.  The last kept one
// is rarely more than ten times below its pivot (the bound is exponential, but not met in practice), so 1e3
// cutoff leaves sqrt(n) and that to spare.  Deciding on pivots alone moved log P of unlikely syndromes by 1e-9
// at the default cutoff (2 of 1500 random networks) and by up to 1e-2 at cutoffs of 1e-3 and above.  In FP32,
// whose rounding is far below the margins (and whose range turns the square of a cutoff below 1e-19 into 0,
// so that only exact zeros are dropped there): point d3, 1 shot 0.755 ms, 0.757 with the squares in FP64.
__device__ __forceinline__ bool cut_rank_decided(double first, double last, double left, int n, double cutoff) {
  const int e = (int)(((unsigned)__double2hiint(first) >> 20) & 0x7FFu) - 1023;
  const float c = cut_f32(cutoff, 0);
  return fabsf(cut_f32(last, e)) > 1e3f * c * fabsf(cut_f32(first, e)) && float(n) * cut_f32(left, 0) <= c * c;
}

// Householder QR with column pivoting of the m x n matrix X (row-major, ld n; destroyed), m <= 64 or so:
// a thread per column, so that every FP64 instruction works on 32 columns (a column per warp leaves
// most lanes idle on the few rows of a cut that does not truncate).  Two barriers per step: pivot;
// reflector (formed by one warp).  Stops at the first pivot norm^2 <= abs2 times that of the first, or after
// `most` steps (*left: the squared norm of the pivot that it stopped at, over the first's); vr[4 j ..]: the
// reflector's head, 2 / v.v, R[j][j] and the pivot column of step j, the reflector's tail in that column; nrm:
// n, keys: nw.
static __device__ __noinline__ int cut_qrcp_cols(Team tm, double* X, int m, int n, double abs2, int most, double* vr,
                                                 double* nrm, unsigned char* taken, unsigned* keys, double& left) {
  const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.nt >> 5, q = m < n ? m : n;
  unsigned best = 0u;
  for (int c = tm.tid; c < n; c += tm.nt) {
    double s = 0.0;
    for (int i = 0; i < m; ++i) s += X[(size_t)i * n + c] * X[(size_t)i * n + c];
    nrm[c] = s;
    taken[c] = 0;
    best = max(best, cut_key(s, c));
  }
  double d02 = 0.0;
  int j = 0;
  left = 0.0;
  for (; j < q; ++j) {
    best = __reduce_max_sync(0xffffffffu, best);
    if (lane == 0) keys[warp] = best;
    tm.sync();
    const unsigned key = cut_best_key(keys, nw, lane);
    if (key == 0u) {
      left = 0.0;
      break;
    }
    const int p = (int)(kCutColMask - (key & kCutColMask));
    const double d2 = nrm[p];
    if (j == 0) d02 = d2;
    left = d02 > 0.0 ? d2 / d02 : 0.0;
    if (!(d2 > 0.0) || d2 <= abs2 * d02 || j >= most) break;
    if (warp == 0) {
      const double x0 = X[(size_t)j * n + p], r = sqrt(d2);
      const double alpha = x0 >= 0.0 ? -r : r;
      const double tau = 1.0 / (d2 + fabs(x0) * r);
      if (lane == 0) {
        vr[4 * j] = x0 - alpha;
        vr[4 * j + 1] = tau;
        vr[4 * j + 2] = alpha;
        vr[4 * j + 3] = double(p);
        taken[p] = 1;
      }
    }
    tm.sync();
    const double v0 = vr[4 * j], tau = vr[4 * j + 1];
    best = 0u;
    for (int c = tm.tid; c < n; c += tm.nt) {
      if (taken[c]) continue;
      const double top = X[(size_t)j * n + c];
      double w = v0 * top;
      for (int i = j + 1; i < m; ++i) w += X[(size_t)i * n + p] * X[(size_t)i * n + c];
      w *= tau;
      double s = 0.0;
      for (int i = j + 1; i < m; ++i) {
        const double x = X[(size_t)i * n + c] - w * X[(size_t)i * n + p];
        X[(size_t)i * n + c] = x;
        s += x * x;
      }
      X[(size_t)j * n + c] = top - w * v0;
      nrm[c] = s;
      best = max(best, cut_key(s, c));
    }
    __syncwarp();
  }
  tm.sync();
  return j;
}

// Cut of rank <= most (nothing to truncate): X = M (m x n, row-major; destroyed); U (m x r) into An
// (row-major), the carry R (r x n) into Cn; Qs: most x m scratch, vr: 4 most, nrm: n, all FP64.  Returns
// r, or -1 when more than `most` pivots lie above the cutoff or the pivots do not decide the rank.
static __device__ __noinline__ int cut_rank(Team tm, double* X, int m, int n, int most, double cutoff, double* An, double* Cn,
                                            double* Qs, double* vr, double* nrm, CutBuf& b, double* s0) {
  double left;
  const int q = m < n ? m : n;
  const int r = cut_qrcp_cols(tm, X, m, n, cutoff * cutoff, most < q ? most : q, vr, nrm, b.taken, b.keys, left);
  if (r == 0) return -1;
  // R[j][j] of the first and the last step
  if (!cut_rank_decided(vr[2], vr[4 * r - 2], r < q ? left : 0.0, n, cutoff)) return -1;
  const int lane = tm.tid & 31, warp = tm.tid >> 5, nw = tm.nt >> 5;
  for (int kk = warp; kk < r; kk += nw) {   // Q e_kk = H_0 ... H_kk e_kk, a warp per column
    double* x = Qs + (size_t)kk * m;
    for (int i = lane; i < m; i += 32) x[i] = i == kk ? 1.0 : 0.0;
    for (int j = kk; j >= 0; --j) {   // a lane's rows are its own: no exchange but the dot product
      const double v0 = vr[4 * j], tau = vr[4 * j + 1];
      const double* v = X + (int)vr[4 * j + 3];
      double w = 0.0;
      for (int i = lane; i < m; i += 32)
        if (i >= j) w += (i == j ? v0 : v[(size_t)i * n]) * x[i];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
      w *= tau;
      for (int i = lane; i < m; i += 32)
        if (i >= j) x[i] -= w * (i == j ? v0 : v[(size_t)i * n]);
    }
  }
  for (int w = tm.tid; w < r * n; w += tm.nt) Cn[w] = X[w];
  tm.sync();
  for (int w = tm.tid; w < r * r; w += tm.nt) {   // pivot columns: alpha on the diagonal, zero below it
    const int j = w / r, i = w % r;
    if (i >= j) Cn[(size_t)i * n + (int)vr[4 * j + 3]] = i == j ? vr[4 * j + 2] : 0.0;
  }
  for (int w = tm.tid; w < m * r; w += tm.nt) An[w] = Qs[(size_t)(w % r) * m + w / r];
  *s0 = fabs(vr[2]);
  tm.sync();
  return r;
}

// Any cut, in FP64: pivoted QR of A (X: n x m scratch), Jacobi on R^T (L, ld cut_ldl); vr: 4 q doubles,
// nrm: max(m, 5 (q + 1) / 2), list: m + q ints (q = min(m, n)); sv: 2 q singular values (unsorted, then
// sorted), ord: their order; slots: four shared ints.  Returns the number kept by the rule (0: the
// matrix is zero or not finite); U into An, the carry into Cn; *rest: the discarded fraction.
static __device__ __noinline__ int cut_full(Team tm, const double* A, int lda, double* X, int m, int n, int most,
                                            double cutoff, double rtol, double* L, double* vr, double* nrm, int* list,
                                            double* sv, int* ord, double* An, double* Cn, CutBuf& b, int* slots,
                                            double* s0, double* rest) {
  const int q = n < m ? n : m;
  for (int w = tm.tid; w < m * n; w += tm.nt) X[w] = A[(size_t)(w % m) * lda + w / m];
  tm.sync();
  double left;
  // directions below 1e-15 of the largest are rounding of A
  const int r = cut_qrcp_cols(tm, X, n, m, 1e-30, q, vr, nrm, b.taken, b.keys, left);
  if (r == 0) return 0;
  const int ldl = cut_ldl(tm.nt, m);
  int* step = list;   // the step in which a column was the pivot
  for (int c = tm.tid; c < m; c += tm.nt) step[c] = r;
  tm.sync();
  for (int j = tm.tid; j < r; j += tm.nt) step[(int)vr[4 * j + 3]] = j;
  tm.sync();
  for (int w = tm.tid; w < r * m; w += tm.nt) {
    const int j = w / m, c = w % m;
    L[(size_t)j * ldl + c] = j < step[c] ? X[w] : (j == step[c] ? vr[4 * j + 2] : 0.0);
  }
  tm.sync();
  if (r > 1) cut_jacobi64(tm, L, ldl, m, r, nrm, list + m, slots);
  cut_order<double>(tm, L, ldl, m, r, sv, ord);
  double* srt = sv + q;
  for (int i = tm.tid; i < r; i += tm.nt) srt[i] = sv[ord[i]];
  tm.sync();
  *s0 = srt[0];
  if (!(srt[0] > 0.0)) return 0;
  if (tm.tid == 0) {
    slots[0] = team_keep_count<double>(srt, r, most, cutoff, rtol);
    double tot = 0.0, disc = 0.0;
    for (int i = 0; i < r; ++i) {
      tot += srt[i] * srt[i];
      if (i >= slots[0]) disc += srt[i] * srt[i];
    }
    b.th[0] = disc / tot;
  }
  tm.sync();
  const int k = slots[0];
  *rest = b.th[0];
  for (int w = tm.tid; w < m * k; w += tm.nt) {
    const int o = ord[w % k];
    An[w] = L[(size_t)o * ldl + w / k] / sv[o];
  }
  tm.sync();
  cut_mul_av(tm, A, lda, n, m, An, k, Cn);
  return k;
}

}  // namespace td
