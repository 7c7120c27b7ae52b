// Simple-update truncation core of one gate (Sec. 4), one team of threads per (gate, shot).
//
// Input: the four Gram blocks G_{X,kappa} (X = A, B; kappa = +, -) of the two sides'
// matrices in the kappa basis of the doubled bond (see sweep.cu).  A pivoted Cholesky
// factor R of each block (G = R^T R, rank-revealing) is an R factor of that side's QR
// decomposition, so the two-site core of the simple update is
//     theta = [c(ka, kb) R_{A ka} Lambda R_{B kb}^T],  c(+,+) = c(-,-) = 1/2,
//     c(+,-) = c(-,+) = (1 - 2p)/2,
// (for the diagonal gate diag(w(r + s_a + s_b)) of the generator picture kappa is the
// physical bit, the blocks are the lo and hi rows themselves and c(ka, kb) = w(r + ka + kb)),
// a (rA x rB) matrix, rA, rB <= 2D.  Its SVD theta = U S V^T is truncated to k <= chi values
// (cutoff and multiplet rule), the bond weight becomes S/s_1 (ln s_1 to the log-scale) and
// the update transforms T_{X kappa} = R_{X kappa}^+ [U or V]_{kappa rows, :k} / sqrt2 are
// written for k_update.
//
// The Gram blocks arrive in FP64 on both paths (summed in FP64 from the stored tensors).
//
// The SVD of theta is FP64 one-sided Jacobi.  With `precond` (the mixed-precision path) it
// is first solved in FP32 on a scaled copy; the FP32 right factor, re-orthogonalised in
// FP64 by one Newton-Schulz step V <- V (3I - V^T V)/2, preconditions the FP64 Jacobi
// sweeps, which are run to convergence (mixed-precision Jacobi: precondition with a
// low-precision factor, finish in high precision).  The FP32 solve cannot resolve singular
// values below ~1e-7 of the largest, and the simple update is sensitive to the ones it keeps
// down to the cutoff, so the FP64 sweeps are not cut short.
#include <cfloat>
#include <cmath>

#include "launch.cuh"
#include "sweep.cuh"
#include "team.cuh"

namespace td {

// Team-shared layout of one item (doubles): five regions of regsz(Dm) = 2Dm x (2Dm + 1)
// (a 2Dm x 2Dm matrix with an odd leading dimension) plus small arrays.
struct CoreSmem {
  double* reg[5];
  double* lam;     // [Dm]
  double* sv;      // [2Dm]
  double* aux;     // [4][Dm] reciprocal Cholesky diagonals, then [2Dm] reciprocal singular values
  int* piv;        // [4][Dm]
  int* order;      // [2Dm]
  int* meta;       // [16]
  static __host__ __device__ size_t regsz(int Dm) { return 4 * (size_t)Dm * Dm + 2 * (size_t)Dm + 2; }
  static __host__ __device__ size_t doubles(int Dm) { return 5 * regsz(Dm) + 7 * (size_t)Dm + 8; }
  static __host__ __device__ size_t ints(int Dm) { return 6 * (size_t)Dm + 16; }
  static __host__ __device__ size_t bytes(int Dm) { return doubles(Dm) * 8 + ints(Dm) * 4 + 16; }
  __device__ void carve(unsigned char* base, int Dm) {
    double* d = reinterpret_cast<double*>(base);
    for (int i = 0; i < 5; ++i) reg[i] = d + (size_t)i * regsz(Dm);
    lam = d + 5 * regsz(Dm);
    sv = lam + Dm;
    aux = sv + 2 * Dm + 8;
    int* ip = reinterpret_cast<int*>(aux + 4 * Dm);
    piv = ip;
    order = piv + 4 * Dm;
    meta = order + 2 * Dm;
  }
};

// The four Gram blocks of item (gate, shot) in FP64: the sum, in chunk order, of the
// partial Grams of its row chunks.
__device__ __forceinline__ void load_gram(const Team& tm, const double* gram, int64_t item, int nchunk, int chi,
                                          int D, double* G) {
  const int DD = D * D;
  const double* src = gram + item * nchunk * 4 * chi * chi;
  for (int w = tm.tid; w < 4 * DD; w += tm.nt) {
    const int64_t off = (int64_t)(w / DD) * chi * chi + w % DD;
    double s = 0.0;
    for (int c = 0; c < nchunk; ++c) s += src[(int64_t)c * 4 * chi * chi + off];
    G[w] = s;
  }
}

// FP64 one-sided Jacobi sweeps (as team_svd_onesided, but V is given and updated) of the items of one block of four
// warps in lock step: up to four items of one-warp teams, two of two, one of four.
//
// What bounds it: an FP64 instruction holds its warp's scheduler for 64 cycles (and the SM's FP64
// pipe for 19) however many lanes are active, so the sweeps cost what their warp instructions cost.  A
// team by itself spends ~93 per step of 8 pairs: 12 for the dot products, 6 for their reduction, ~43
// for the test and the rotation's angles (division, square roots; the same in the 4 lanes of a pair),
// 32 to apply it -- also for pairs that do not rotate.  Here one warp computes the angles of all the
// block's pairs, one pair per lane, and the rotations of the pairs that rotate are spread over all
// four warps row by row; a pair's three sums are reduced side by side (3 instead of 6 instructions for
// 4 lanes), or, when a block has fewer items than warps, by different warps.  The same operations in
// the same order on every value: bit for bit the result of team_svd_onesided.  Measured (core time of
// a decode, before -> with this; the angles' quotients in integers, ieee.cuh, took off another 6-11 %):
// rotated d9 chi 8, 1000 shots mixed 178 -> 129 ms, 152 shots FP64 66 -> 47 ms; d7 FP64, 48 shots
// 29.4 -> 18.9 ms; d5, 37 shots 10.1 -> 7.4 ms.
// Not done: keeping the squared norms of columns that did not rotate (a twelfth fewer FP64 instructions):
// 121.5 -> 120.5 ms with a full chip, but 6.8 -> 7.2 ms for d5, 37 shots, where a step is a chain.
struct GroupJacobi {
  double al[32], be[32], ga[32];   // squared norms and inner product of every pair of the step
  double c[32], s[32];
  int pq[32];                      // p | q << 8 | valid << 16 | parity of the item's sweep << 17
  int list[32];                    // slots of the pairs that rotate
  int cnt;
  int any[4][2];                   // a rotation in the item's sweep (by the sweep's parity)
  double *A[4], *V[4];
  int lda[4], ldv[4], m[4], n[4];
};
constexpr int kGroupBar = 15;
// Items per SM below which a round's blocks take fewer items than they have teams for.  Measured
// (core time of a decode, ms, at 0 / 4 / 8 / 16 / 32): rotated d5 chi 8, 37 shots 9.7 / 7.4 / 7.4 / 7.4 / 7.4,
// 300 shots 11.5 / 11.5 / 10.9 / 11.2 / 11.3; rotated d7 FP64, 48 shots 26.2 / 23.0 / 18.9 / 18.9 / 18.9;
// rotated d9 FP64, 152 shots 47.4 / 47.4 / 47.4 / 50.3 / 59.6.
constexpr int kCoreSpread = 8;

__device__ __forceinline__ bool group_sync_or(bool p) {
  int r;
  __syncwarp();   // the barrier takes whole warps
  asm volatile(
      "{\n.reg .pred a, b;\nsetp.ne.s32 a, %1, 0;\nbar.red.or.pred b, %2, 128, a;\nselp.s32 %0, 1, 0, b;\n}\n"
      : "=r"(r)
      : "r"((int)p), "n"(kGroupBar)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void group_sync() {
  __syncwarp();
  asm volatile("bar.sync %0, 128;" ::"n"(kGroupBar) : "memory");
}

// items: of the block (4, 2 or 1); nt: threads of a team, the first of an item's 128 / items threads;
// the item's arrays are given by its team's thread 0 (has: it has a matrix to work on).
__device__ void group_jacobi(GroupJacobi& gj, int items, int nt, bool has, double* A, int lda, int m, int n, double* V,
                             int ldv, int max_sweeps) {
  const int gt = threadIdx.x, gw = gt >> 5, lane = gt & 31;
  const int per = 128 / items, it = gt / per, ti = gt % per;
  const int subs = per / nt, sub = ti / nt, tid = ti % nt;
  const int S = nt / 4;   // pair slots per item
  if (ti == 0) {
    gj.A[it] = A;
    gj.V[it] = V;
    gj.lda[it] = lda;
    gj.ldv[it] = ldv;
    gj.m[it] = m;
    gj.n[it] = has && n >= 2 ? n : 0;
    gj.any[it][0] = gj.any[it][1] = 0;
  }
  if (gt < 32) gj.pq[gt] = 0;
  if (!group_sync_or(ti == 0 && has && n >= 2)) return;
  A = gj.A[it];
  lda = gj.lda[it];
  m = gj.m[it];
  n = gj.n[it];
  bool busy = n > 0;
  int R = 0;   // rows of the block's largest rotation
  for (int i = 0; i < items; ++i)
    if (gj.n[i] > 0) R = max(R, gj.m[i] + gj.n[i]);
  const int ne = n + (n & 1), half = ne / 2;
  int g = half > 0 ? nt / half : 1;        // lanes per pair, as team_svd_onesided
  g = g < 1 ? 1 : (g > 32 ? 32 : team_pow2_floor(g));
  const int rows_max = m > n ? m : n;
  while (g > 1 && g > rows_max) g >>= 1;
  const int grp = tid / g, gl = tid % g;
  int k = 0, sweep = 0, turn = 0;
  for (;;) {
    // the step's inner products
    if (ti < S) {
      int p, q;
      team_rr_pair(k, ti, ne, p, q);
      gj.pq[it * S + ti] = (busy && ti < half && q < n) ? (p | q << 8 | 1 << 16 | (sweep & 1) << 17) : 0;
    }
    if (k == 0 && ti == 0) gj.any[it][(sweep & 1) ^ 1] = 0;   // read before the last barrier
    if (busy) {
      int p = 0, q = 0;
      bool active = grp < half;
      if (active) {
        team_rr_pair(k, grp, ne, p, q);
        active = q < n;
      }
      const double* ap_ = A + (size_t)p * lda;
      const double* aq_ = A + (size_t)q * lda;
      const int slot = it * S + grp;
      if (subs == 1) {
        double al = 0.0, be = 0.0, ga = 0.0;
        if (active)
          for (int r = gl; r < m; r += g) {
            const double ap = ap_[r], aq = aq_[r];
            al += ap * ap;
            be += aq * aq;
            ga += ap * aq;
          }
        // sums over the pair's lanes, offsets g/2, g/4, ..., 1: the upper half of the lanes takes be, the
        // lower al, both ga; from the second level on every lane sums one value
        if (g >= 2) {
          const bool up = (gl & (g >> 1)) != 0;
          const double other = __shfl_xor_sync(0xffffffffu, up ? al : be, g >> 1);
          const double og = __shfl_xor_sync(0xffffffffu, ga, g >> 1);
          double v = (up ? be : al) + other;
          ga += og;
          if (g >= 4) {
            const bool up2 = (gl & (g >> 2)) != 0;
            const double o2 = __shfl_xor_sync(0xffffffffu, up2 ? v : ga, g >> 2);
            v = (up2 ? ga : v) + o2;
            for (int o = g >> 3; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (active) {
              if (gl == 0) gj.al[slot] = v;
              else if (gl == (g >> 2)) gj.ga[slot] = v;
              else if (gl == (g >> 1)) gj.be[slot] = v;
            }
          } else if (active) {
            if (up) {
              gj.be[slot] = v;
            } else {
              gj.al[slot] = v;
              gj.ga[slot] = ga;
            }
          }
        } else if (active) {
          gj.al[slot] = al;
          gj.be[slot] = be;
          gj.ga[slot] = ga;
        }
      } else {
        // spare warps: the sums by different ones (two: al and be | ga; four: one each)
        for (int f = sub; f < 3; f += subs) {   // f: 0 al, 1 ga, 2 be
          double v = 0.0;
          const double* x = f == 2 ? aq_ : ap_;
          const double* y = f == 0 ? ap_ : aq_;
          if (active)
            for (int r = gl; r < m; r += g) v += x[r] * y[r];
          for (int o = g >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (active && gl == 0) (f == 0 ? gj.al : f == 1 ? gj.ga : gj.be)[slot] = v;
        }
      }
    }
    group_sync();
    // angles: one pair per lane, the warps in turn
    if (gw == turn) {
      const int pq = gj.pq[lane];
      double c = 1.0, s = 0.0;
      bool act = false;
      if (pq) act = jacobi_rot(gj.al[lane], gj.be[lane], gj.ga[lane], TeamTol<double>::rel(), c, s);
      const unsigned mask = __ballot_sync(0xffffffffu, act);
      if (act) {
        gj.c[lane] = c;
        gj.s[lane] = s;
        gj.list[__popc(mask & ((1u << lane) - 1u))] = lane;
        gj.any[lane / S][(pq >> 17) & 1] = 1;
      }
      if (lane == 0) gj.cnt = __popc(mask);
    }
    turn = (turn + 1) & 3;
    group_sync();
    // rotations: the rows of the pairs that rotate, A's then V's, over the block's threads
    const int tasks = gj.cnt * R;
    for (int t = gt; t < tasks; t += 128) {
      const int e = t / R, r = t - e * R;
      const int slot = gj.list[e], i = slot / S, pq = gj.pq[slot];
      const int mi = gj.m[i], p = pq & 255, q = (pq >> 8) & 255;
      if (r < mi + gj.n[i]) {
        const bool inA = r < mi;
        double* base = inA ? gj.A[i] : gj.V[i];
        const int ld = inA ? gj.lda[i] : gj.ldv[i], row = inA ? r : r - mi;
        double* xp = base + (size_t)p * ld + row;
        double* xq = base + (size_t)q * ld + row;
        const double c = gj.c[slot], s = gj.s[slot];
        const double ap = *xp, aq = *xq;
        *xp = c * ap - s * aq;
        *xq = s * ap + c * aq;
      }
    }
    if (busy && ++k == ne - 1) {
      const int any = gj.any[it][sweep & 1];
      k = 0;
      if (!any || ++sweep == max_sweeps) busy = false;
    }
    if (!group_sync_or(busy)) break;
  }
}

__global__ void k_core2(SweepArgs a, const GateDesc* __restrict__ gates, const double* __restrict__ gram,
                        double* __restrict__ tbuf, int S, int n_items, int items, int team_threads, int Dm, int precond) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ GroupJacobi gj;
  // `items` items per block of 128 threads; an item's first team_threads threads are its team, the
  // rest only help in the group's Jacobi sweeps
  const int per = 128 / items, team = threadIdx.x / per;
  const int64_t item = (int64_t)blockIdx.x * items + team;
  if (item >= n_items || (int)threadIdx.x % per >= team_threads) {
    group_jacobi(gj, items, team_threads, false, nullptr, 1, 0, 0, nullptr, 1, 40);
    return;
  }
  Team tm;
  tm.nt = team_threads;
  tm.tid = threadIdx.x % per;
  tm.bar = 1 + team;
  CoreSmem sm;
  sm.carve(smem_raw + (size_t)team * CoreSmem::bytes(Dm), Dm);
  const int gi = (int)(item / a.B), b = (int)(item % a.B);
  const GateDesc& gd = gates[gi];
  const int D = gd.D, Dn = gd.Dn, chi = a.chi, DD = D * D;
  int* meta = sm.meta;
  double* slot = reinterpret_cast<double*>(sm.sv + 2 * Dm);   // one spare double after sv
  double* RG = sm.reg[0];
  double* RF = sm.reg[1];
  double* RI = sm.reg[2];
  double* TH = sm.reg[3];
  double* VV = sm.reg[4];
  load_gram(tm, gram, item, a.gram_chunks, chi, D, RG);
  double* lamg = a.lam + ((int64_t)b * a.nbonds + gd.bond) * chi;
  for (int w = tm.tid; w < D; w += tm.nt) sm.lam[w] = lamg[w];
  tm.sync();
  // pivot tolerance per block: gram_cutoff times the side's largest diagonal (< 0: empty)
  if (tm.tid < 4) {
    const int side = tm.tid / 2;
    long long top = 0;   // on the bit patterns: NaN above infinity above the finite values, negative ones below 0
    for (int blk = 2 * side; blk < 2 * side + 2; ++blk)
      for (int j = 0; j < D; ++j) top = max(top, __double_as_longlong(RG[blk * DD + j * D + j]));
    const double e = __longlong_as_double(top);
    if (non_finite(e)) mark_non_finite(a, b);
    sm.sv[tm.tid] = e > 0.0 ? a.gram_cutoff * e : -1.0;
  }
  tm.sync();
  int* rkp = meta + 12;
  team_pchol4(tm, RG, D, DD, sm.sv, RF, sm.piv, sm.aux, Dm, rkp);
  team_pchol_rinv4(tm, RF, D, DD, sm.piv, sm.aux, Dm, rkp, RI);
  int rk[4];
  for (int blk = 0; blk < 4; ++blk) rk[blk] = rkp[blk];
  double* Rm = RF;           // R factor rows (r x D, ld D) per block
  const double* Rinv = RI;   // right inverse (D x r, ld D) per block
  double* FF = RG;           // scratch free during the SVD (the Gram is consumed)
  double* TT = RF;           // scratch free once theta is formed (R is consumed)
  const int rAp = rk[0], rA = rk[0] + rk[1], rBp = rk[2], rB = rk[2] + rk[3];
  double* tout = tbuf + item * 4 * chi * chi;
  // record for the reverse sweep: ranks, old lambda, R factors and right inverses
  double* rec = a.rec_core ? a.rec_core + ((int64_t)(a.gate_base + gi - a.rec_gate0) * a.B + b) * core_rec_elems(chi)
                           : nullptr;
  const int CC = chi * chi, L2 = 2 * chi;
  if (rec) {
    if (tm.tid < 4) rec[tm.tid] = rk[tm.tid];
    if (tm.tid == 4) { rec[4] = 0.0; rec[5] = 0.0; }
    for (int w = tm.tid; w < D; w += tm.nt) rec[8 + w] = sm.lam[w];
    for (int w = tm.tid; w < 4 * DD; w += tm.nt) {
      rec[8 + chi + (w / DD) * CC + w % DD] = RF[w];
      rec[8 + chi + 4 * CC + (w / DD) * CC + w % DD] = RI[w];
    }
  }
  if (rA == 0 || rB == 0) {            // zero state: this shot has probability 0
    for (int w = tm.tid; w < 4 * chi * chi; w += tm.nt) tout[w] = 0.0;
    for (int w = tm.tid; w < Dn; w += tm.nt) lamg[w] = 0.0;
    if (tm.tid == 0) a.logacc[(int64_t)b * a.nslots + S + gd.bond] = -INFINITY;
    group_jacobi(gj, items, team_threads, false, nullptr, 1, 0, 0, nullptr, 1, 40);
    return;
  }
  const Override* ov = vshot_ovr(a.vs, a.ovr, a.wave_first, b, kOvrGate, a.gate_base + gi);
  const double p = ov ? ov->val[0] : gd.p;
  // core coefficients c(ka, kb): kappa = +/- for the gate (1-p) I x I + p X x X; for the
  // diagonal gate of the generator picture kappa is the physical bit itself and
  // c(ka, kb) = w(r + ka + kb), w = (1-p, p), with r the shot's bit of the gate's qubit
  double c_eq = 0.5, c_ne = 0.5 * (1.0 - 2.0 * p);
  if (gd.diag) {
    const int r = a.det[(int64_t)vshot_row(a.vs, a.wave_first, b) * a.n_det + gd.rcol] & 1;
    c_eq = r ? p : 1.0 - p;
    c_ne = r ? 1.0 - p : p;
  }
  for (int w = tm.tid; w < rA * D; w += tm.nt) {     // R_A Lambda, in place
    const int i = w / D, q = w % D;
    const int ka = i < rAp ? 0 : 1, li = i - ka * rAp;
    Rm[ka * DD + li * D + q] *= sm.lam[q];
  }
  tm.sync();
  // theta[i][j] = c(ki, kj) sum_q (R_{A ki} Lambda)[li][q] R_{B kj}[lj][q]  (column-major)
  const int ldt = odd_ld(rA), ldv = odd_ld(rB);
  for (int w = tm.tid; w < rA * rB; w += tm.nt) {
    const int j = w / rA, i = w % rA;
    const int ka = i < rAp ? 0 : 1, li = i - ka * rAp;
    const int kb = j < rBp ? 0 : 1, lj = j - kb * rBp;
    const double* ra = Rm + ka * DD + li * D;
    const double* rb = Rm + (2 + kb) * DD + lj * D;
    double s = 0.0;
    for (int q = 0; q < D; ++q) s += ra[q] * rb[q];
    TH[j * ldt + i] = (ka == kb ? c_eq : c_ne) * s;
  }
  tm.sync();
  if (precond)
    svd_precond(tm, TH, ldt, rA, rB, VV, ldv, FF, TT, meta + 8, slot);
  else
    for (int w = tm.tid; w < rB * rB; w += tm.nt) VV[(w / rB) * ldv + (w % rB)] = (w / rB == w % rB) ? 1.0 : 0.0;
  tm.sync();
  group_jacobi(gj, items, team_threads, true, TH, ldt, rA, rB, VV, ldv, 40);
  tm.sync();
  team_col_norms<double>(tm, TH, ldt, rA, rB, sm.sv);
  team_sort_desc<double>(tm, sm.sv, rB, sm.order);
  if (tm.tid == 0) {
    double srt[2 * kMaxChi];
    for (int j = 0; j < rB; ++j) srt[j] = sm.sv[sm.order[j]];
    int k = 0;
    if (srt[0] > 0.0) k = team_keep_count<double>(srt, rB < rA ? rB : rA, Dn, a.svd_cutoff, a.multiplet_rtol);
    meta[0] = k;
    if (a.stats && k > 0) {
      // discarded fraction sum_{j >= k} s_j^2 / sum_j s_j^2; the shot's gates of a round run
      // concurrently: the max on the bit patterns (non-negative doubles order as them)
      double tot = 0.0, disc = 0.0;
      for (int j = 0; j < rB; ++j) {
        const double q = srt[j] * srt[j];
        tot += q;
        if (j >= k) disc += q;
      }
      const double f = tot > 0.0 ? disc / tot : 0.0;
      double* st = a.stats + (int64_t)(a.wave_first + b) * 4;
      atomicMax(reinterpret_cast<unsigned long long*>(st), (unsigned long long)__double_as_longlong(f));
      atomicAdd(st + 1, f);
    }
  }
  tm.sync();
  const int k = meta[0];
  const double s0 = sm.sv[sm.order[0]];
  if (k == 0 || !(s0 > 0.0)) {
    for (int w = tm.tid; w < 4 * chi * chi; w += tm.nt) tout[w] = 0.0;
    for (int w = tm.tid; w < Dn; w += tm.nt) lamg[w] = 0.0;
    if (tm.tid == 0) {
      a.logacc[(int64_t)b * a.nslots + S + gd.bond] = -INFINITY;
      if (non_finite(s0)) mark_non_finite(a, b);
    }
    return;
  }
  if (rec) {
    double* rUS = rec + 8 + chi + 8 * CC;
    double* rV = rUS + L2 * L2;
    double* rsv = rV + L2 * L2;
    double* rord = rsv + L2;
    for (int w = tm.tid; w < rA * rB; w += tm.nt) rUS[(w / rA) * L2 + w % rA] = TH[(w / rA) * ldt + w % rA];
    for (int w = tm.tid; w < rB * rB; w += tm.nt) rV[(w / rB) * L2 + w % rB] = VV[(w / rB) * ldv + w % rB];
    for (int w = tm.tid; w < rB; w += tm.nt) { rsv[w] = sm.sv[w]; rord[w] = sm.order[w]; }
    if (tm.tid == 0) { rec[4] = k; rec[5] = s0; }
  }
  for (int j = tm.tid; j < k; j += tm.nt) sm.aux[j] = 1.0 / sm.sv[sm.order[j]];
  tm.sync();
  const double rs2 = gd.diag ? 1.0 : 0.70710678118654752440;   // the kappa basis' 1/sqrt2
  // T_{A kap}[q][j] = sum_{li} R^+_{A kap}[q][li] U[kap rows li][order j] / sqrt2, U = theta_out / s
  for (int w = tm.tid; w < 2 * D * Dn; w += tm.nt) {
    const int kap = w / (D * Dn), q = (w / Dn) % D, j = w % Dn;
    double acc = 0.0;
    if (j < k) {
      const int cj = sm.order[j];
      const int r = rk[kap], off = kap ? rAp : 0;
      const double* ri = Rinv + kap * DD + q * D;
      const double* u = TH + cj * ldt + off;
      for (int li = 0; li < r; ++li) acc += ri[li] * u[li];
      acc *= sm.aux[j];
    }
    tout[(int64_t)kap * chi * chi + q * Dn + j] = acc * rs2;
  }
  for (int w = tm.tid; w < 2 * D * Dn; w += tm.nt) {
    const int kap = w / (D * Dn), q = (w / Dn) % D, j = w % Dn;
    double acc = 0.0;
    if (j < k) {
      const int cj = sm.order[j];
      const int r = rk[2 + kap], off = kap ? rBp : 0;
      const double* ri = Rinv + (2 + kap) * DD + q * D;
      const double* v = VV + cj * ldv + off;
      for (int lj = 0; lj < r; ++lj) acc += ri[lj] * v[lj];
    }
    tout[(int64_t)(2 + kap) * chi * chi + q * Dn + j] = acc * rs2;
  }
  const double is0 = sm.aux[0];
  for (int j = tm.tid; j < Dn; j += tm.nt) lamg[j] = (j < k) ? sm.sv[sm.order[j]] * is0 : 0.0;
  if (tm.tid == 0) a.logacc[(int64_t)b * a.nslots + S + gd.bond] += log(s0);
}

// ---- launch configuration ---------------------------------------------------------------
// Blocks of 128 threads.  Team by bond dimension: one warp, two or four (four segments of at least
// Dm lanes for the four Cholesky factorisations).  Items per block: as many as there are teams when
// the round fills the chip; fewer when it does not, so that an item has spare warps on the other
// schedulers and the blocks reach more SMs.
static int core_team(int Dm) { return Dm <= 8 ? 32 : (Dm <= 16 ? 64 : 128); }

template <typename R>
cudaError_t launch_core2(const SweepArgs& a, const GateDesc* g, int count, int Dm, const double* gram, double* tbuf,
                         int S, bool precond, cudaStream_t st) {
  const int tt = core_team(Dm);
  const int64_t n_items = (int64_t)count * a.B;
  int dev = 0, nsm = 1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  int items = 128 / tt;
  while (items > 1 && n_items <= (int64_t)kCoreSpread * nsm * items / 4) items /= 2;
  const size_t smem = (size_t)items * CoreSmem::bytes(Dm);
  e = allow_shared_memory<k_core2>();
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)((n_items + items - 1) / items);
  k_core2<<<blocks, 128, smem, st>>>(a, g, gram, tbuf, S, (int)n_items, items, tt, Dm, precond ? 1 : 0);
  return cudaGetLastError();
}

template cudaError_t launch_core2<double>(const SweepArgs&, const GateDesc*, int, int, const double*, double*, int,
                                          bool, cudaStream_t);
template cudaError_t launch_core2<float>(const SweepArgs&, const GateDesc*, int, int, const double*, double*, int,
                                         bool, cudaStream_t);

}  // namespace td
