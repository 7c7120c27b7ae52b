// Team-cooperative dense linear algebra for the small FP64/FP32 factorisations of the
// sweep (Sec. 4 simple-update truncation) and of the final boundary-MPS contraction.
//
// A team is a group of nt threads of one block (nt = 32: one warp, synchronised with
// __syncwarp; nt a larger multiple of 32: its own named barrier).  Several teams share a
// block, each working on an independent problem, so no step waits on a block-wide barrier.
//
// Methods (textbook, written for this layout):
//   * pivoted Cholesky of a positive semi-definite Gram matrix (Golub & Van Loan,
//     Matrix Computations, 4th ed., Alg. 4.2.4 with diagonal pivoting, Sec. 4.2.8), stopped
//     at the first pivot below a tolerance: a rank-revealing R factor of the Gram's matrix;
//   * the inverse of the triangular part by back substitution (ibid. Sec. 3.1);
//   * the one-sided (Hestenes) Jacobi SVD with the round-robin parallel ordering
//     (ibid. Sec. 8.6.3 and 8.5.5): the n/2 column pairs of one step are disjoint, so each
//     pair is handled by its own group of g lanes, which computes the pair's three inner
//     products (lane partial sums combined by shuffles), the rotation (the symmetric 2x2
//     Schur rotation, ibid. Alg. 8.5.1), and applies it to both columns of A and of V.
//     One barrier per step.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "finlayout.cuh"
#include "ieee.cuh"

namespace td {

struct Team {
  int tid;   // thread index inside the team
  int nt;    // team size: 32, or a multiple of 32 using named barrier `bar`
  int bar;   // named barrier id (1..15), unused for nt == 32
  __device__ __forceinline__ void sync() const {
    if (nt == 32)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(nt) : "memory");
  }
};

template <typename R>
struct TeamTol;
template <>
struct TeamTol<double> {
  static __device__ __forceinline__ double rel() { return 1e-15; }
  static __device__ __forceinline__ double tiny() { return 1e-290; }
};
template <>
struct TeamTol<float> {
  static __device__ __forceinline__ float rel() { return 1e-7f; }
  static __device__ __forceinline__ float tiny() { return 1e-30f; }
};

// Pair i of step k of the round-robin ("circle") ordering of ne (even) players; player
// ne-1 stays in place.  p < q on return.
__device__ __forceinline__ void team_rr_pair(int k, int i, int ne, int& p, int& q) {
  const int m = ne - 1;   // 0 <= k < m, 0 <= i < ne / 2
  p = k + i;
  if (p >= m) p -= m;
  q = k - i;
  if (q < 0) q += m;
  if (i == 0) q = m;
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
}

// Four independent pivoted Cholesky factorisations of symmetric positive semi-definite D x D blocks run
// concurrently: the team is split into four lane segments of seg = nt/4 lanes (D <= seg <= 32); segment b
// factors the block G + b*bstride (row-major, destroyed) into Rf + b*bstride (ld D).  Pivot k is the largest
// remaining diagonal entry; the factorisation stops when it is <= tol[b] (< 0 marks an empty block, rank 0).
// Rows 0..r-1 of the factor are in the original column order -- G ~= Rf^T Rf, Rf[i][piv[j]] = 0 for j < i --,
// the pivot columns and the reciprocals of R11's diagonal (from one rsqrt per pivot) in piv/dinv + b*pstride,
// the rank in rank[b] (team-shared).  Pivot
// candidates are compared as bit patterns: non-negative doubles order as integers, and a
// negative rounding residue loses to any admissible pivot.
__device__ __forceinline__ void team_pchol4(const Team& tm, double* G, int D, int bstride, const double* tol,
                                            double* Rf, int* piv, double* dinv, int pstride, int* rank) {
  const int seg = tm.nt / 4;
  const int blk = tm.tid / seg, sl = tm.tid % seg;
  double* Gb = G + blk * bstride;
  double* Rb = Rf + blk * bstride;
  const double tl = tol[blk];
  const long long tbits = __double_as_longlong(tl);
  bool active = tl >= 0.0;
  uint32_t done = 0;
  int r = 0;
  for (int k = 0; k < D; ++k) {
    long long key = -1;
    int idx = sl;
    if (active && sl < D && !((done >> sl) & 1u)) key = __double_as_longlong(Gb[sl * D + sl]);
    for (int o = seg >> 1; o > 0; o >>= 1) {
      const long long k2 = __shfl_xor_sync(0xffffffffu, key, o);
      const int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
      if (k2 > key || (k2 == key && i2 < idx)) {
        key = k2;
        idx = i2;
      }
    }
    const bool ok = active && key > tbits;
    const int p = idx;
    if (ok) {
      const double dpp = Gb[p * D + p];
      const double inv = rsqrt(dpp);
      const double rkk = dpp * inv;
      for (int c = sl; c < D; c += seg) {
        double v;
        if (c == p)
          v = rkk;
        else if ((done >> c) & 1u)
          v = 0.0;
        else
          v = Gb[p * D + c] * inv;
        Rb[k * D + c] = v;
      }
      if (sl == 0) {
        piv[blk * pstride + k] = p;
        dinv[blk * pstride + k] = inv;
      }
      done |= 1u << p;
      r = k + 1;
    } else {
      active = false;
    }
    tm.sync();
    if (ok)
      for (int w = sl; w < D * D; w += seg) {
        const int a = w / D, c = w % D;
        if (((done >> a) & 1u) || ((done >> c) & 1u)) continue;
        Gb[a * D + c] -= Rb[k * D + a] * Rb[k * D + c];
      }
    tm.sync();
  }
  if (sl == 0) rank[blk] = r;
  tm.sync();
}

// Right inverses of the four factors of team_pchol4: Ri + b*bstride is D x r_b (ld D) with Rf Ri = 1, nonzero
// only in the pivot rows: Ri[piv[i]][j] = (R11^-1)[i][j], R11[i][j] = Rf[i][piv[j]] upper triangular, by back
// substitution with the stored reciprocal diagonals; one (block, column) per thread.
__device__ __forceinline__ void team_pchol_rinv4(const Team& tm, const double* Rf, int D, int bstride, const int* piv,
                                                 const double* dinv, int pstride, const int* rank, double* Ri) {
  for (int w = tm.tid; w < 4 * D * D; w += tm.nt) Ri[(w / (D * D)) * bstride + w % (D * D)] = 0.0;
  tm.sync();
  const int seg = tm.nt / 4;
  const int blk = tm.tid / seg, j = tm.tid % seg;
  const int r = rank[blk];
  if (j < r) {
    const double* Rb = Rf + blk * bstride;
    double* Ib = Ri + blk * bstride;
    const int* pb = piv + blk * pstride;
    const double* db = dinv + blk * pstride;
    Ib[pb[j] * D + j] = db[j];
    for (int i = j - 1; i >= 0; --i) {
      double s = 0.0;
      for (int l = i + 1; l <= j; ++l) s += Rb[i * D + pb[l]] * Ib[pb[l] * D + j];
      Ib[pb[i] * D + j] = -s * db[i];
    }
  }
  tm.sync();
}

// Comparisons of the Jacobi test on bit patterns where the values are known not to be negative (they
// order as integers): an FP64 comparison holds the FP64 pipe like a multiplication.  le: a <= b for
// a, b >= 0 (false when either is NaN, as in floating point).
__device__ __forceinline__ bool nonneg_le(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return x <= y && y <= 0x7FF0000000000000ll;
}
__device__ __forceinline__ bool nonneg_le(float a, float b) { return a <= b; }
__device__ __forceinline__ bool is_zero(double a) { return (__double_as_longlong(a) << 1) == 0ll; }
__device__ __forceinline__ bool is_zero(float a) { return a == 0.f; }
__device__ __forceinline__ bool below_zero(double a) { return __double_as_longlong(a) < 0ll && !is_zero(a); }
__device__ __forceinline__ bool below_zero(float a) { return a < 0.f; }

// Rotation (c, s) of the one-sided Jacobi step for columns with squared norms al, be and
// inner product ga; false when the pair is already orthogonal to working precision
// (ga^2 <= tol^2 al be), or when a column is negligible (squared norm below tiny(); FP32
// solves run on matrices scaled to a largest entry of 1).  In FP64 the quotients and the root are formed
// in integer arithmetic (ieee.cuh): 15 FP64 instructions instead of 40, the same values.
template <typename R>
__device__ __forceinline__ bool jacobi_rot(R al, R be, R ga, R tol, R& c, R& s) {
  if (is_zero(ga) || nonneg_le(al, TeamTol<R>::tiny()) || nonneg_le(be, TeamTol<R>::tiny()) ||
      nonneg_le(ga * ga, tol * tol * (al * be))) {
    c = R(1);
    s = R(0);
    return false;
  }
  const R zeta = ieee_div(be - al, R(2) * ga);
  const R t = ieee_div(below_zero(zeta) ? R(-1) : R(1), fabs(zeta) + ieee_sqrt(R(1) + zeta * zeta));
  c = rsqrt(R(1) + t * t);
  s = t * c;
  return true;
}

// Largest power of two <= x (x >= 1).
__device__ __forceinline__ int team_pow2_floor(int x) {
  int g = 1;
  while (2 * g <= x) g *= 2;
  return g;
}

// One-sided Jacobi SVD of the m x n matrix A, stored column-major (element (r, c) at
// A[c * lda + r]; an odd lda keeps the lanes of different column pairs on different shared
// memory banks): on return the columns of A are mutually orthogonal, A_out = A_in V, with
// V (n x n, column-major, ldv) orthogonal -- so the singular values are the column norms
// of A_out and its normalised columns the left singular vectors.  `flag` is one int of
// team-shared scratch.  Returns the number of sweeps.
template <typename R>
__device__ int team_svd_onesided(const Team& tm, R* A, int lda, int m, int n, R* V, int ldv, int* flag,
                                 int max_sweeps) {
  const R tol = TeamTol<R>::rel();
  for (int w = tm.tid; w < n * n; w += tm.nt) V[(w / n) * ldv + (w % n)] = (w / n == w % n) ? R(1) : R(0);
  tm.sync();
  if (n < 2) return 0;
  const int ne = n + (n & 1), half = ne / 2;
  int g = tm.nt / half;
  g = g < 1 ? 1 : (g > 32 ? 32 : team_pow2_floor(g));
  const int rows_max = m > n ? m : n;
  while (g > 1 && g > rows_max) g >>= 1;
  const int ngroups = tm.nt / g;
  const int grp = tm.tid / g, gl = tm.tid % g;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (tm.tid == 0) *flag = 0;
    tm.sync();
    for (int k = 0; k < ne - 1; ++k) {
      for (int i0 = 0; i0 < half; i0 += ngroups) {
        const int i = i0 + grp;
        int p = 0, q = 0;
        bool active = i < half;
        if (active) {
          team_rr_pair(k, i, ne, p, q);
          active = q < n;
        }
        R* ap_ = A + (size_t)p * lda;
        R* aq_ = A + (size_t)q * lda;
        R al = R(0), be = R(0), ga = R(0);
        if (active)
          for (int r = gl; r < m; r += g) {
            const R ap = ap_[r], aq = aq_[r];
            al += ap * ap;
            be += aq * aq;
            ga += ap * aq;
          }
        for (int o = g >> 1; o > 0; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o);
          be += __shfl_xor_sync(0xffffffffu, be, o);
          ga += __shfl_xor_sync(0xffffffffu, ga, o);
        }
        R c, s;
        if (active && jacobi_rot(al, be, ga, tol, c, s)) {
          if (gl == 0) *flag = 1;
          for (int r = gl; r < m; r += g) {
            const R ap = ap_[r], aq = aq_[r];
            ap_[r] = c * ap - s * aq;
            aq_[r] = s * ap + c * aq;
          }
          R* vp_ = V + (size_t)p * ldv;
          R* vq_ = V + (size_t)q * ldv;
          for (int r = gl; r < n; r += g) {
            const R vp = vp_[r], vq = vq_[r];
            vp_[r] = c * vp - s * vq;
            vq_[r] = s * vp + c * vq;
          }
        }
      }
      tm.sync();
    }
    const int any = *flag;
    tm.sync();
    if (!any) break;
  }
  return sweep;
}

// Column norms of A (m x n, column-major, lda): out[j] = ||A[:, j]||.
template <typename R>
__device__ void team_col_norms(const Team& tm, const R* A, int lda, int m, int n, R* out) {
  for (int j = tm.tid; j < n; j += tm.nt) {
    const R* a = A + (size_t)j * lda;
    R s = R(0);
    for (int r = 0; r < m; ++r) s += a[r] * a[r];
    out[j] = sqrt(s);
  }
  tm.sync();
}

// Odd leading dimension >= rows (column-major storage without bank-aligned columns).
__host__ __device__ __forceinline__ int odd_ld(int rows) { return rows | 1; }

// Descending order of n non-negative values (ties: lower index first): order[rank] = j.
// Ranks are counted on the bit patterns, which order non-negative IEEE values exactly.
template <typename R>
__device__ void team_sort_desc(const Team& tm, const R* v, int n, int* order) {
  for (int j = tm.tid; j < n; j += tm.nt) {
    const double vj = double(v[j]);
    const long long bj = __double_as_longlong(vj);
    int rank = 0;
    for (int i = 0; i < n; ++i) {
      const long long bi = __double_as_longlong(double(v[i]));
      rank += (bi > bj || (bi == bj && i < j)) ? 1 : 0;
    }
    order[rank] = j;
  }
  tm.sync();
}

// Number of singular values kept: s (descending, s[0] > 0); at most chi, only those above
// cutoff * s[0]; a cut inside a multiplet (s[k-1] - s[k] <= rtol * s[0]) drops it whole
// unless that leaves nothing.
template <typename R>
__device__ __forceinline__ int team_keep_count(const R* s, int n, int chi, double cutoff, double rtol) {
  int r = 0;
  while (r < n && double(s[r]) > cutoff * double(s[0])) ++r;
  int k = r < chi ? r : chi;
  if (k < r) {
    int kk = k;
    while (kk > 0 && double(s[kk - 1]) - double(s[kk]) <= rtol * double(s[0])) --kk;
    if (kk > 0) k = kk;
  }
  return k;
}

// Max |x| over the m x n column-major matrix x (ld), through a shared double slot.
__device__ inline double team_absmax(const Team& tm, const double* x, int ld, int m, int n, double* slot) {
  // on the bit patterns, which order non-negative doubles (an FP64 fmax is two FP64 instructions); a
  // NaN does not count, as in fmax
  unsigned long long v = 0ull;
  for (int w = tm.tid; w < m * n; w += tm.nt) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(x[(w / m) * ld + (w % m)]) & 0x7FFFFFFFFFFFFFFFull;
    v = (u > v && u <= 0x7FF0000000000000ull) ? u : v;
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
    v = u > v ? u : v;
  }
  if (tm.tid == 0) *slot = 0.0;
  tm.sync();
  if ((tm.tid & 31) == 0) atomicMax(reinterpret_cast<unsigned long long*>(slot), v);
  tm.sync();
  const double r = *slot;
  tm.sync();
  return r;
}

// Start of a one-sided Jacobi SVD of A (m x n, column-major, lda) from an FP32 solve
// (mixed-precision Jacobi): the FP32 Jacobi runs on a copy scaled to a largest entry of 1; its
// right factor, re-orthogonalised in FP64 by one Newton-Schulz step V <- V (3I - V^T V) / 2, is applied
// to A in FP64; FP64 Jacobi sweeps (the caller's, V updated along) then run to convergence from it.
// The FP32 solve cannot resolve singular values below ~1e-7 of the largest, so the FP64 sweeps are
// never cut short.  V column-major (ldv).  F: scratch of >= max(m, n) * (max(m, n) + 1) doubles (it
// also holds the two FP32 matrices); Tt: >= n*n doubles; flag: one team-shared int; slot: one
// team-shared double.  Not synchronised on return.
__device__ inline void svd_precond(const Team& tm, double* A, int lda, int m, int n, double* V, int ldv, double* F,
                                   double* Tt, int* flag, double* slot) {
  const double amax = team_absmax(tm, A, lda, m, n, slot);
  if (!(amax > 0.0) || n < 2) {   // nothing to precondition: V = 1
    for (int w = tm.tid; w < n * n; w += tm.nt) V[(w / n) * ldv + (w % n)] = (w / n == w % n) ? 1.0 : 0.0;
    return;
  }
  const int la32 = odd_ld(m), lv32 = odd_ld(n);
  float* A32 = reinterpret_cast<float*>(F);
  float* V32 = A32 + la32 * n;
  const double sc = 1.0 / amax;
  for (int w = tm.tid; w < m * n; w += tm.nt) {
    const int c = w / m, r = w % m;
    A32[c * la32 + r] = float(A[c * lda + r] * sc);
  }
  tm.sync();
  team_svd_onesided<float>(tm, A32, la32, m, n, V32, lv32, flag, 30);
  for (int w = tm.tid; w < n * n; w += tm.nt) {
    const int c = w / n, r = w % n;
    V[c * ldv + r] = double(V32[c * lv32 + r]);
  }
  tm.sync();
  // Newton-Schulz: V <- V (3I - V^T V) / 2   (Tt, F: column-major, ld n); V^T V is
  // symmetric: the entries i <= j are computed and mirrored (the same products in the same
  // order, so the mirror is exact)
  for (int w = tm.tid; w < n * (n + 1) / 2; w += tm.nt) {
    int j = (int)((sqrtf(8.0f * w + 1.0f) - 1.0f) * 0.5f);   // corrected below
    while ((j + 1) * (j + 2) / 2 <= w) ++j;
    while (j * (j + 1) / 2 > w) --j;
    const int i = w - j * (j + 1) / 2;   // 0 <= i <= j
    const double* vi = V + i * ldv;
    const double* vj = V + j * ldv;
    double s = 0.0;
    for (int l = 0; l < n; ++l) s += vi[l] * vj[l];
    const double t = (i == j ? 1.5 : 0.0) - 0.5 * s;
    Tt[j * n + i] = t;
    Tt[i * n + j] = t;
  }
  tm.sync();
  for (int w = tm.tid; w < n * n; w += tm.nt) {
    const int j = w / n, i = w % n;
    double s = 0.0;
    for (int l = 0; l < n; ++l) s += V[l * ldv + i] * Tt[j * n + l];
    F[j * n + i] = s;
  }
  tm.sync();
  for (int w = tm.tid; w < n * n; w += tm.nt) V[(w / n) * ldv + (w % n)] = F[w];
  tm.sync();
  // A <- A V   (F: column-major, ld m)
  for (int w = tm.tid; w < m * n; w += tm.nt) {
    const int j = w / m, i = w % m;
    double s = 0.0;
    for (int l = 0; l < n; ++l) s += A[l * lda + i] * V[j * ldv + l];
    F[j * m + i] = s;
  }
  tm.sync();
  for (int w = tm.tid; w < m * n; w += tm.nt) A[(w / m) * lda + (w % m)] = F[w];
}

}  // namespace td
