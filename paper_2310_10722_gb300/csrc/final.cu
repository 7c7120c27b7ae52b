// Final 2D contraction (Sec. 4: "the remaining two-dimensional network is contracted by
// sweeping an MPS across it"; chi_MPS of Sec. 5) and the coset log-sum / decision.
//
// Site tensor of the final network: F[c][l][r][d][u] = sum_phys R[phys][c] Gamma[phys][..]
// with sqrt(lambda) absorbed on every bond; c is the site's class bit.  Rows y = 0..ny-1 are
// absorbed into a boundary MPS A_x[a][d][b] by zip-up: a carry C[j][a][l][p] runs left to
// right, T[j][u][b][r][q] = sum C A F~ with F~[l,p; r,q] = F[p^q], and (j,u) x (b,r,q) is
// truncated to chi_mps by its leading singular vectors.  The class parity p flows along
// each row into a two-valued output leg of the last MPS tensor.  The last row is contracted
// exactly.
//
// Arithmetic.  The contraction computes in FP64 on both paths (T is the storage type of the
// site tensors it reads): the class-parity leg carries both cosets through one MPS, so FP32
// sums and FP32 singular vectors err by ~eps32 times the majority coset's weight, a relative
// error of ~eps32 exp(margin) on the minority coset.  The cuts are those of cut.cuh, to FP64
// accuracy on every path; the gradient pass's recorded forward takes a one-sided Jacobi SVD of
// M^T with V accumulated (its records are M^T V and V), with the rounding of team_svd_onesided for a block
// of that size: the adjoint divides by differences of singular values, so another rounding here moves single
// entries of the gradient by up to 1e-6.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "cut.cuh"
#include "launch.cuh"
#include "sweep.cuh"
#include "team.cuh"

namespace td {

// F[c][l][r][d][u] of site (x, y) into F (dims into fd: L, R, D, U; fd[4] = 1 when the
// class-1 half F[1] can be nonzero, 0 when it is exactly zero -- the readout has no class
// flip).  sqrt(lambda) of the site's bonds is staged in slam[4][chi] first.
template <typename T, typename R>
__device__ void build_F(const Team& tm, const FinalArgs& fa, int b, int x, int y, R* F, int* fd, R* slam) {
  const int s = fa.grid_site[y * fa.nx + x];
  if (s < 0) {
    if (tm.tid == 0) { F[0] = R(1); F[1] = R(0); fd[4] = 0; }
    if (tm.tid < 4) fd[tm.tid] = 1;
    tm.sync();
    return;
  }
  const FinalSite& fs = fa.sites[s];
  const Override* ov = vshot_ovr(fa.vs, fa.ovr, fa.wave_first, b, kOvrRead, s);
  const double* Rv = ov ? ov->val : fs.R;
  const double* lam = fa.lam + (int64_t)b * fa.nbonds * fa.chi;
  for (int w = tm.tid; w < 4 * fa.chi; w += tm.nt) {
    const int dir = w / fa.chi, i = w % fa.chi;
    slam[w] = (fs.dir_pos[dir] >= 0 && i < fs.dir_dim[dir]) ? R(sqrt(lam[fs.dir_bond[dir] * fa.chi + i])) : R(1);
  }
  const int dL = fs.dir_dim[0], dR = fs.dir_dim[1], dD = fs.dir_dim[2], dU = fs.dir_dim[3];
  int stride[4];   // stride of each direction's index in the site tensor (0 if absent)
  {
    int st[kMaxBonds];
    int acc = 1;
    for (int k = fs.nb - 1; k >= 0; --k) {
      st[k] = acc;
      int dk = 1;
      for (int dir = 0; dir < 4; ++dir)
        if (fs.dir_pos[dir] == k) dk = fs.dir_dim[dir];
      acc *= dk;
    }
    for (int dir = 0; dir < 4; ++dir) stride[dir] = fs.dir_pos[dir] >= 0 ? st[fs.dir_pos[dir]] : 0;
  }
  const int rest = dL * dR * dD * dU;
  const T* g = reinterpret_cast<const T*>(fa.gamma) + (int64_t)b * fa.shot_elems + fs.off;
  tm.sync();
  for (int w = tm.tid; w < rest; w += tm.nt) {
    int e = w;
    const int iu = e % dU; e /= dU;
    const int id = e % dD; e /= dD;
    const int ir = e % dR; e /= dR;
    const int il = e;
    const int off = il * stride[0] + ir * stride[1] + id * stride[2] + iu * stride[3];
    const R wgt = slam[il] * slam[fa.chi + ir] * slam[2 * fa.chi + id] * slam[3 * fa.chi + iu];
    R a0 = R(0), a1 = R(0);
    for (int ph = 0; ph < fs.P; ++ph) {
      const R gv = R(g[(int64_t)ph * rest + off]);
      a0 += R(Rv[ph * 2 + 0]) * gv;
      a1 += R(Rv[ph * 2 + 1]) * gv;
    }
    F[w] = a0 * wgt;
    F[rest + w] = a1 * wgt;
  }
  if (tm.tid == 0) {
    fd[0] = dL; fd[1] = dR; fd[2] = dD; fd[3] = dU;
    int c1 = 0;
    for (int ph = 0; ph < fs.P; ++ph) c1 |= (Rv[ph * 2 + 1] != 0.0);
    fd[4] = c1;
  }
  tm.sync();
}

// Discarded fraction of a cut: |M - U U^T M|^2 over |M|^2, entry by entry (no cancellation); M = MT^T, U (m x k,
// row-major), C = U^T M (k x n).
static __device__ __noinline__ double cut_discarded(Team tm, const double* MT, int ldm, int m, int n, const double* U,
                                                    const double* C, int k, double (*sums)[32]) {
  double disc = 0.0, tot = 0.0;
  for (int w = tm.tid; w < m * n; w += tm.nt) {
    const int c = w / n, i = w % n;
    const double a = MT[(size_t)c * ldm + i];
    double d = a;
    for (int j = 0; j < k; ++j) d -= C[(size_t)j * n + i] * U[c * k + j];
    disc += d * d;
    tot += a * a;
  }
  for (int o = 16; o > 0; o >>= 1) {
    disc += __shfl_xor_sync(0xffffffffu, disc, o);
    tot += __shfl_xor_sync(0xffffffffu, tot, o);
  }
  if ((tm.tid & 31) == 0) {
    sums[0][tm.tid >> 5] = disc;
    sums[1][tm.tid >> 5] = tot;
  }
  tm.sync();
  disc = tot = 0.0;
  for (int w = 0; w < tm.nt / 32; ++w) {
    disc += sums[0][w];
    tot += sums[1][w];
  }
  return disc / tot;
}

// The cut of M = MT^T (m x n) by cut.cuh: the left vectors into An, the unscaled
// carry into Cn.  Returns the number of states kept (0: the matrix is zero, or *s0 says not finite), or -1
// when the scratch does not hold the paths (the caller then takes the plain Jacobi of the recorded cuts).
// Scratch: shared memory (`pool` bytes at `sp`) as far as it goes, then the W, Q and R regions.
static __device__ __noinline__ int cut(Team tm, const FinalArgs& fa, const double* MT, int ldm, int m, int n,
                                       double* work, double* W, double* An, double* Cn, unsigned char* sp, int64_t pool,
                                       int* slots, double (*sums)[32], double* trunc, double* s0) {
  const int q = m < n ? m : n, cm = fa.chi_mps, kk = cm < q ? cm : q;
  const int ex = cut_max_exponent(tm, MT, ldm, n, m, slots) - 1023;
  *s0 = ldexp(1.0, ex);   // infinite for an infinity or NaN in the matrix (ex = 1024)
  if (ex == -1023 || ex == 1024) return 0;
  if (m == 1) {
    // one state (outside the occupied grid): U = 1, carry = M
    for (int w = tm.tid; w < n; w += tm.nt) Cn[w] = MT[w];
    if (tm.tid == 0) An[0] = 1.0;
    return 1;
  }
  CutBuf cb;
  int64_t wleft = fa.W_elems * 8;
  unsigned char* wp = reinterpret_cast<unsigned char*>(W);
  const int64_t small = CutBuf::small_bytes(m, n, kk);
  if (small <= pool) {
    cb.carve_small(sp, m, n, kk);
    sp += small;
    pool -= small;
  } else if (small <= wleft) {
    cb.carve_small(wp, m, n, kk);
    wp += small;
    wleft -= small;
  } else {
    return -1;
  }
  double* Q = work + fa.w_Q;
  double* Rg = work + fa.w_R;
  const int64_t l_col = 4 * (int64_t)cut_ld32(tm.nt, m);   // bytes of an FP32 column
  int k = -1, r32 = 0;
  double rest = 0.0;   // discarded fraction
  if (q > cm && ex > -400 && ex < 400) {
    r32 = q;
    const int64_t vec_p = CutBuf::vec_bytes(m, n, cm, true), vec = CutBuf::vec_bytes(m, n, cm, false);
    const bool vs = vec_p + l_col * q <= pool;
    if (vs || vec <= wleft) {
      if (vs) cb.carve_vec(reinterpret_cast<double*>(sp), m, n, cm, nullptr);
      else cb.carve_vec(reinterpret_cast<double*>(wp), m, n, cm, Cn);
      unsigned char* lp = vs ? sp + vec_p : sp;
      const int64_t cap = (vs ? pool - vec_p : pool) / 4;
      if (cut_topk(tm, MT, ldm, n, m, cm, fa.svd_cutoff, fa.multiplet_rtol, ex, reinterpret_cast<float*>(Q),
                   reinterpret_cast<float*>(Rg), reinterpret_cast<float*>(lp), (int)cap, cb, slots, s0, &r32)) {
        k = cm;
        for (int w = tm.tid; w < m * k; w += tm.nt) An[w] = cb.V[w];
        if (vs)
          for (int w = tm.tid; w < k * n; w += tm.nt) Cn[w] = cb.P[w];
        if (fa.stats) rest = cut_discarded(tm, MT, ldm, m, n, cb.V, cb.P, k, sums);
      }
    }
  }
  if (k < 0 && r32 <= cm) {
    const int64_t need_v = 8 * (4 * (int64_t)kk + n), need_q = 8 * (int64_t)kk * m, need_x = 8 * (int64_t)m * n;
    if (need_v + need_q <= wleft) {
      const bool xs = need_v + need_q + need_x <= pool;
      unsigned char* base = xs ? sp : wp;
      double* vr = reinterpret_cast<double*>(base);
      double* nrm = vr + 4 * kk;
      double* Qs = nrm + n;
      double* X = xs ? Qs + (size_t)kk * m : Q;
      for (int w = tm.tid; w < m * n; w += tm.nt) X[w] = MT[(size_t)(w / n) * ldm + w % n];
      tm.sync();
      k = cut_rank(tm, X, m, n, kk, fa.svd_cutoff, An, Cn, Qs, vr, nrm, cb, s0);
      if (fa.stats && k > 0 && k < q) rest = cut_discarded(tm, MT, ldm, m, n, An, Cn, k, sums);
    }
  }
  if (k < 0) {
    const int ints = (m + q + 1) & ~1, nb = m > 5 * (q + 1) / 2 ? m : 5 * (q + 1) / 2;
    const int64_t need_v = 8 * (4 * (int64_t)q + nb) + 4 * ints, need_l = 8 * (int64_t)cut_ldl(tm.nt, m) * q,
                  need_x = 8 * (int64_t)m * n;
    const bool vs = need_v <= pool;
    if (vs || need_v <= wleft) {
      double* vr = reinterpret_cast<double*>(vs ? sp : wp);
      double* nrm = vr + 4 * q;
      int* list = reinterpret_cast<int*>(nrm + nb);
      if (vs) {
        sp += (need_v + 15) / 16 * 16;
        pool -= (need_v + 15) / 16 * 16;
      }
      const bool ls = need_l <= pool, xs = need_l + need_x <= pool;
      double* L = ls ? reinterpret_cast<double*>(sp) : Rg;
      double* X = xs ? reinterpret_cast<double*>(sp + need_l) : Q;
      k = cut_full(tm, MT, ldm, X, m, n, cm, fa.svd_cutoff, fa.multiplet_rtol, L, vr, nrm, list, work + fa.w_s,
                   reinterpret_cast<int*>(work + fa.w_ord), An, Cn, cb, slots, s0, &rest);
    }
  }
  if (k > 0 && fa.stats && tm.tid == 0) {
    trunc[0] = fmax(trunc[0], rest);
    trunc[1] += rest;
  }
  tm.sync();
  return k;
}

// One block per shot.  The work region (site tensor F, T1 / V, M^T, carries) lives in
// shared memory when it fits, otherwise in the shot's global scratch; the boundary MPS is
// always in global scratch.
// NT: threads per block; MINB: resident blocks that the registers are to leave room for.
template <typename T, typename R, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_final(FinalArgs fa) {
  const int b = blockIdx.x;
  const Team tm{(int)threadIdx.x, (int)blockDim.x, 1};
  extern __shared__ __align__(16) unsigned char smem_raw[];
  R* scr = reinterpret_cast<R*>(fa.scratch) + (int64_t)b * fa.scratch_elems;
  R* work = fa.use_smem ? reinterpret_cast<R*>(smem_raw) : scr + fa.off_work;
  R* mps[2] = {scr + fa.off_mps0, scr + fa.off_mps1};
  R* F = work + fa.w_F;
  R* W = work + fa.w_W;        // T1, then V of the SVD
  R* MT = work + fa.w_MT;      // M^T (n x m)
  R* Cb[2] = {work + fa.w_C0, work + fa.w_C1};
  R* sv = work + fa.w_s;
  int* ord = reinterpret_cast<int*>(work + fa.w_ord);
  __shared__ int mdim[2][kMaxGridX][3];   // per column: (left, down, right) of the MPS tensors
  __shared__ int fd[5];
  __shared__ int meta[8];
  __shared__ R slam[4 * kMaxChi];
  __shared__ double logsum_s;
  __shared__ double trunc_s[2];   // largest and summed discarded fraction of the cuts
  __shared__ double sum_s[2][32];
  const int nx = fa.nx, ny = fa.ny;
  if (isnan(fa.logacc[(int64_t)b * fa.nslots + fa.slot])) {   // mark_non_finite
    if (tm.tid < 2) fa.Z[(int64_t)b * 2 + tm.tid] = NAN;
    return;
  }
  if (tm.tid == 0) { logsum_s = 0.0; trunc_s[0] = 0.0; trunc_s[1] = 0.0; }
  for (int x = tm.tid; x < nx; x += tm.nt) {
    mdim[0][x][0] = 1; mdim[0][x][1] = 1; mdim[0][x][2] = (x == nx - 1) ? 2 : 1;
    R* A = mps[0] + (int64_t)x * fa.mps_stride;
    A[0] = R(1);
    if (x == nx - 1) A[1] = R(0);
  }
  tm.sync();
  int cur = 0;
  for (int y = 0; y < ny; ++y) {
    int cc = 0;
    if (tm.tid == 0) { Cb[0][0] = R(1); Cb[0][1] = R(0); }
    int cJ = 1, cA = 1, cL = 1;
    tm.sync();
    for (int x = 0; x < nx; ++x) {
      build_F<T, R>(tm, fa, b, x, y, F, fd, slam);
      const int L = fd[0], Rr = fd[1], U = fd[3];
      const R* A = mps[cur] + (int64_t)x * fa.mps_stride;
      const int aL = mdim[cur][x][0], aD = mdim[cur][x][1], aR = mdim[cur][x][2];
      const R* C = Cb[cc];
      (void)cA;
      // T1[l][p][d][bb][j] = sum_a C[j][a][l][p] A[a][d][bb]  (j fastest: the lanes of one
      // warp below read four j values of the same (l, p, d, bb) from distinct banks)
      double* rs = nullptr;    // this column's record slot (reverse sweep)
      if constexpr (sizeof(R) == 8) {
        if (fa.rec) {
          rs = fa.rec + (int64_t)b * fa.rec_stride + (int64_t)(y * nx + x) * fa.rec_slot;
          const FinRecSlot ly(fa.rec_mC, fa.rec_mA, fa.rec_m, fa.rec_n);
          for (int w = tm.tid; w < cJ * aL * cL * 2; w += tm.nt) rs[ly.C + w] = double(C[w]);
          for (int w = tm.tid; w < aL * aD * aR; w += tm.nt) rs[ly.A + w] = double(A[w]);
          if (tm.tid == 0) {
            rs[1] = cJ; rs[2] = aL; rs[3] = cL; rs[4] = aD; rs[5] = aR;
            rs[6] = L; rs[7] = Rr; rs[8] = U;
            rs[0] = (x == nx - 1) ? 2 : (y == ny - 1 ? 1 : 0);
          }
        }
      }
      R* T1 = W;
      const int n1 = cJ * L * 2 * aD * aR;
      for (int w = tm.tid; w < n1; w += tm.nt) {
        int e = w;
        const int j = e % cJ; e /= cJ;
        const int bb = e % aR; e /= aR;
        const int d = e % aD; e /= aD;
        const int p = e % 2; e /= 2;
        const int l = e;
        R acc = R(0);
        for (int a = 0; a < aL; ++a) acc += C[((j * aL + a) * cL + l) * 2 + p] * A[(a * aD + d) * aR + bb];
        T1[w] = acc;
      }
      tm.sync();
      // MT[(bb, r, q)][(j, u)] = sum_{l,p,d} T1[l][p][d][bb][j] F[p^q][l][r][d][u], stored
      // column-major: column (j, u) of MT is row (j, u) of M; leading dimensions chosen so
      // the Jacobi lane groups of consecutive columns fall on disjoint banks where they fit
      const int nF = L * Rr * aD * U;
      const int m = cJ * U, n = aR * Rr * 2;
      const int pc = fd[4];   // 0: F[1] is zero, so only p = q contributes (half the products)
      const int lanes = team_svd_group(tm.nt, n, m);
      const int ldm = final_ld(n, lanes, m, fa.MT_elems), ldv = final_ld(m, lanes, m, fa.W_elems);
      for (int w = tm.tid; w < m * n; w += tm.nt) {
        const int c = w / m, ju = w % m;      // consecutive lanes: consecutive u (F) and ju (MT)
        const int q = c % 2, r = (c / 2) % Rr, bb = c / (2 * Rr);
        const int j = ju / U, u = ju % U;
        R acc = R(0);
        const int p_lo = pc ? 0 : q, p_hi = pc ? 2 : q + 1;
        for (int l = 0; l < L; ++l)
          for (int p = p_lo; p < p_hi; ++p) {
            const R* t1 = T1 + (((l * 2 + p) * aD) * aR + bb) * cJ + j;
            const R* f = F + (p ^ q) * nF + ((l * Rr + r) * aD) * U + u;
            for (int d = 0; d < aD; ++d) acc += t1[d * aR * cJ] * f[d * U];
          }
        MT[ju * ldm + c] = acc;
      }
      tm.sync();
      R* An = mps[cur ^ 1] + (int64_t)x * fa.mps_stride;
      R* Cn = Cb[cc ^ 1];
      if (x < nx - 1 && y < ny - 1) {
        int k = -1;   // states kept; -1: by the plain Jacobi below
        double s0 = 0.0;
        if constexpr (sizeof(R) == 8) {
          if (!rs)
            k = cut(tm, fa, MT, ldm, m, n, work, W, An, Cn, smem_raw + (fa.use_smem ? fa.work_elems * sizeof(R) : 0),
                    fa.cut_smem, meta + 2, sum_s, trunc_s, &s0);
        }
        R* V = W;
        const bool plain = k < 0;
        if (plain) {
          // one-sided Jacobi on the m columns of MT, V accumulated (the reverse sweep's record)
          if constexpr (sizeof(R) == 8) {
            const int half = (m + 1) / 2;
            if (24 * half * 2 <= fa.cut_smem) {   // 5 doubles and an int per pair
              double* buf = reinterpret_cast<double*>(smem_raw + (fa.use_smem ? fa.work_elems * sizeof(R) : 0));
              block_svd_onesided(tm, MT, ldm, n, m, V, ldv, buf, reinterpret_cast<int*>(buf + 5 * half), meta + 2, 40);
            } else {
              team_svd_onesided<R>(tm, MT, ldm, n, m, V, ldv, meta + 7, 40);
            }
          }
          team_col_norms<R>(tm, MT, ldm, n, m, sv);
          team_sort_desc<R>(tm, sv, m, ord);
          if (tm.tid == 0) {
            int kept = 0;
            if (sv[ord[0]] > R(0)) {
              R* srt = sv + m;   // the second half of the singular-value region
              const int nsv = m < n ? m : n;
              for (int i = 0; i < nsv; ++i) srt[i] = sv[ord[i]];
              kept = team_keep_count<R>(srt, nsv, fa.chi_mps, fa.svd_cutoff, fa.multiplet_rtol);
              if (fa.stats) {   // discarded fraction sum_{i >= k} s_i^2 / sum_i s_i^2
                double tot = 0.0, disc = 0.0;
                for (int i = 0; i < nsv; ++i) {
                  const double q = double(srt[i]) * double(srt[i]);
                  tot += q;
                  if (i >= kept) disc += q;
                }
                const double f = tot > 0.0 ? disc / tot : 0.0;
                trunc_s[0] = fmax(trunc_s[0], f);
                trunc_s[1] += f;
              }
            }
            meta[0] = kept;
          }
          tm.sync();
          k = meta[0];
          s0 = double(sv[ord[0]]);
        }
        if constexpr (sizeof(R) == 8) {
          if (rs) {
            const FinRecSlot ly(fa.rec_mC, fa.rec_mA, fa.rec_m, fa.rec_n);
            for (int w = tm.tid; w < m * m; w += tm.nt) rs[ly.V + w] = double(V[(w / m) * ldv + w % m]);
            for (int w = tm.tid; w < n * m; w += tm.nt) rs[ly.MT + w] = double(MT[(w / n) * ldm + w % n]);
            for (int w = tm.tid; w < m; w += tm.nt) { rs[ly.sv + w] = double(sv[w]); rs[ly.ord + w] = ord[w]; }
            if (tm.tid == 0) {
              int e2r = 0;
              if (k > 0) frexp(s0, &e2r);
              rs[9] = m; rs[10] = n; rs[11] = k; rs[12] = e2r;
            }
          }
        }
        if (k == 0) {
          if (tm.tid == 0) logsum_s += non_finite(s0) ? NAN : -INFINITY;
          for (int w = tm.tid; w < m; w += tm.nt) An[w] = R(0);
          for (int w = tm.tid; w < n; w += tm.nt) Cn[w] = R(0);
          if (tm.tid == 0) { mdim[cur ^ 1][x][0] = cJ; mdim[cur ^ 1][x][1] = U; mdim[cur ^ 1][x][2] = 1; }
          cJ = 1;
        } else {
          // exact power-of-two normalisation of the carry (its log to the log-scale)
          int e2 = 0;
          frexp(s0, &e2);
          const R inv0 = R(ldexp(1.0, -e2));
          if (plain) {
            for (int w = tm.tid; w < m * k; w += tm.nt) {
              const int ju = w / k, kk = w % k;
              An[w] = V[ord[kk] * ldv + ju];
            }
            for (int w = tm.tid; w < k * n; w += tm.nt) {
              const int kk = w / n, c = w % n;
              Cn[w] = MT[ord[kk] * ldm + c] * inv0;
            }
          } else {
            for (int w = tm.tid; w < k * n; w += tm.nt) Cn[w] *= inv0;
          }
          if (tm.tid == 0) {
            logsum_s += double(e2) * 0.69314718055994530942;
            mdim[cur ^ 1][x][0] = cJ; mdim[cur ^ 1][x][1] = U; mdim[cur ^ 1][x][2] = k;
          }
          cJ = k;
        }
        cA = aR; cL = Rr;
        cc ^= 1;
        tm.sync();
      } else if (x < nx - 1) {
        // last row: U == 1, no truncation; the carry takes the whole contraction
        if (rs && tm.tid == 0) { rs[9] = m; rs[10] = n; }
        for (int w = tm.tid; w < m * n; w += tm.nt) {
          const int ju = w / n, c = w % n;
          Cn[w] = MT[ju * ldm + c];
        }
        for (int w = tm.tid; w < m * m; w += tm.nt) An[w] = (w / m == w % m) ? R(1) : R(0);
        if (tm.tid == 0) { mdim[cur ^ 1][x][0] = cJ; mdim[cur ^ 1][x][1] = U; mdim[cur ^ 1][x][2] = m; }
        cJ = m; cA = aR; cL = Rr;
        cc ^= 1;
        tm.sync();
      } else {
        // last column (Rr == 1): merge the old class leg bb and the row parity q into bb ^ q
        for (int w = tm.tid; w < m * 2; w += tm.nt) {
          const int ju = w / 2, c2 = w % 2;
          R acc = R(0);
          for (int bb = 0; bb < aR; ++bb) acc += MT[ju * ldm + bb * 2 + (bb ^ c2)];
          An[w] = acc;
        }
        tm.sync();
        if (tm.tid < 32) {
          R mx = R(0);
          for (int w = tm.tid; w < m * 2; w += 32) mx = fmax(mx, fabs(An[w]));
          for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
          if (tm.tid == 0) {
            meta[1] = 0;
            int e2 = 0;
            if (mx > R(0)) {
              frexp(double(mx), &e2);
              logsum_s += double(e2) * 0.69314718055994530942;
            } else {
              logsum_s += -INFINITY;
            }
            slam[0] = mx > R(0) ? R(ldexp(1.0, -e2)) : R(0);
            if (rs) { rs[9] = m; rs[10] = n; rs[12] = e2; }
            mdim[cur ^ 1][x][0] = cJ; mdim[cur ^ 1][x][1] = U; mdim[cur ^ 1][x][2] = 2;
          }
        }
        tm.sync();
        const R inv = slam[0];
        if (inv > R(0))
          for (int w = tm.tid; w < m * 2; w += tm.nt) An[w] *= inv;
        tm.sync();
      }
    }
    cur ^= 1;
    tm.sync();
  }
  // contract the last MPS (vertical legs are trivial): v <- v A_x, the vectors in the two
  // carry buffers (each holds at least chi_mps * final bond dimension values)
  {
    R* v = Cb[0];
    R* vn = Cb[1];
    if (tm.tid == 0) v[0] = R(1);
    int dv = 1;
    tm.sync();
    for (int x = 0; x < nx; ++x) {
      const R* A = mps[cur] + (int64_t)x * fa.mps_stride;
      const int aL = mdim[cur][x][0], aR = mdim[cur][x][2];
      const int na = aL < dv ? aL : dv;
      for (int bb = tm.tid; bb < aR; bb += tm.nt) {
        R acc = R(0);
        for (int a = 0; a < na; ++a) acc += v[a] * A[a * aR + bb];
        vn[bb] = acc;
      }
      tm.sync();
      R* t = v; v = vn; vn = t;
      dv = aR;
    }
    if (tm.tid == 0) {
      fa.Z[(int64_t)b * 2 + 0] = double(v[0]);
      fa.Z[(int64_t)b * 2 + 1] = double(v[1]);
      fa.logacc[(int64_t)b * fa.nslots + fa.slot] = logsum_s;
      if (fa.stats) {
        fa.stats[(int64_t)(fa.wave_first + b) * 4 + 2] = trunc_s[0];
        fa.stats[(int64_t)(fa.wave_first + b) * 4 + 3] = trunc_s[1];
      }
    }
  }
}

__global__ void k_finalize(FinalizeArgs f) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= f.B) return;
  double ls = 0.0;
  for (int k = 0; k < f.nslots; ++k) ls += f.logacc[(int64_t)b * f.nslots + k];
  const double z0 = f.Z[2 * b], z1 = f.Z[2 * b + 1];
  double zz[2] = {f.mix[0] * z0 + f.mix[1] * z1, f.mix[2] * z0 + f.mix[3] * z1};
  int off = 0;
  if (f.offset_all) {
    const uint8_t* m = f.det + (int64_t)vshot_row(f.vs, f.wave_first, b) * f.n_det;
    for (int i = 0; i < f.n_det; ++i) off ^= m[i] & 1;
  }
  double lp[2];
  for (int c = 0; c < 2; ++c) {
    const double z = zz[c ^ off];
    lp[c] = (z > 0.0 && ls > -INFINITY) ? log(z) + ls : -INFINITY;
  }
  // a non-finite intermediate (NaN in a log-scale or in the final contraction, or an
  // infinite weight) makes the shot's result NaN and is reported by td_network_check
  if (isnan(ls) || isnan(z0) || isnan(z1) || ls == INFINITY || isinf(z0) || isinf(z1)) {
    lp[0] = lp[1] = NAN;
    if (f.status) atomicExch(f.status, (int)TD_ERR_NUMERIC);
  }
  const int64_t gb = f.wave_first + b;
  if (f.logp) {
    f.logp[2 * gb] = lp[0];
    f.logp[2 * gb + 1] = lp[1];
  }
  const int dec = (lp[1] > lp[0]) ? 1 : 0;
  if (f.decision) f.decision[gb] = dec;
  if (f.margin) f.margin[gb] = lp[dec] - lp[dec ^ 1];
}

template <typename T, typename R, int NT, int MINB>
static cudaError_t final_launch(const FinalArgs& f, cudaStream_t st) {
  FinalArgs a = f;
  // dynamic shared memory: the work region when it fits, then scratch for the cuts -- what the
  // largest can use, within the share of an SM that leaves room for as many blocks as there are (at
  // most MINB)
  int dev = 0, nsm = 1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int64_t wk = f.use_smem ? f.work_elems * (int64_t)sizeof(R) : 0;
  const int per_sm = std::max(1, std::min(MINB, (f.B + nsm - 1) / nsm));
  const int64_t room = std::min<int64_t>(f.smem_block, f.smem_sm / per_sm - 1024) - (int64_t)kFinalStaticSmem - wk;
  const int64_t pool = std::max<int64_t>(0, std::min<int64_t>(room, f.rec ? 48 * (f.rec_m + 2) / 2 : f.cut_need)) / 16 * 16;
  a.cut_smem = (int32_t)pool;
  const size_t smem = (size_t)(wk + pool);
  if (smem > 0) {
    e = allow_shared_memory<k_final<T, R, NT, MINB>>();
    if (e != cudaSuccess) return e;
  }
  k_final<T, R, NT, MINB><<<f.B, NT, smem, st>>>(a);
  return cudaGetLastError();
}

template <typename T, typename R>
cudaError_t launch_final(const FinalArgs& f, cudaStream_t st) {
  switch (f.threads) {
    case 256: return final_launch<T, R, 256, 3>(f, st);
    case 512: return final_launch<T, R, 512, 1>(f, st);
    default: return final_launch<T, R, 1024, 1>(f, st);
  }
}

cudaError_t launch_finalize(const FinalizeArgs& f, cudaStream_t st) {
  k_finalize<<<(f.B + 127) / 128, 128, 0, st>>>(f);
  return cudaGetLastError();
}

// ---- final contraction with scratch in a static device array ----------------------------
// For callers that cannot call cudaMalloc: the scratch of k_final comes from this
// file-scope array instead of the network workspace.  Every GPU that loads the library holds
// it until the process exits.  Host code must not use the symbol as an address; the device
// address is looked up once per device (cudaGetSymbolAddress) with that device current.
static __device__ __align__(256) unsigned char g_final_scratch[kStaticFinalScratchBytes];

namespace {
std::mutex g_static_mu;
void* g_static_ptr[kMaxStaticDevices] = {};
}  // namespace

cudaError_t static_final_scratch(void** ptr) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxStaticDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_final_scratch);
    if (e != cudaSuccess) return e;
    g_static_ptr[dev] = p;
  }
  *ptr = g_static_ptr[dev];
  return cudaSuccess;
}

template cudaError_t launch_final<double, double>(const FinalArgs&, cudaStream_t);
template cudaError_t launch_final<float, double>(const FinalArgs&, cudaStream_t);

}  // namespace td
