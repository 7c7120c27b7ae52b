// Layer absorption of the boundary sweep (Sec. 4) on the GPU: site-local operators, and
// for every two-site gate (1-p) I x I + p X x X on a bond (the natural split of Sec. 5.1)
// the simple-update truncation of that bond back to chi (Sec. 4): Gram pass (absorb.cu),
// truncation core (core.cu), update pass (absorb.cu).
//
// Gate as bond doubling: with k the gate's bit, Gamma'_X[sigma; ..., (b, k)] =
// Gamma_X[sigma ^ k mask_X; ..., b] and lambda'_(b,k) = lambda_b w_k, w = (1-p, p).  In the
// basis kappa = (k=0 +- k=1)/sqrt2 the Gram matrix of M'_X (Gamma'_X with the other bonds'
// lambdas absorbed) is block diagonal: G+ = sum Y Y^T, G- = sum Z Z^T over rows, where
// Y = M[sigma_lo] + M[sigma_hi], Z = M[sigma_lo] - M[sigma_hi] for each pair
// sigma_hi = sigma_lo ^ mask.  The core kernel turns the four blocks into R factors,
// forms the 2D x 2D core theta = R_A Lambda' R_B^T, takes its SVD and keeps <= chi values;
// the update applies Gamma_new[lo] = Y T+ + Z T-, Gamma_new[hi] = Y T+ - Z T-.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "sweep.cuh"

namespace td {

template <typename T>
__global__ void k_init(SweepArgs a, const LocalDesc* __restrict__ locals0, int S) {
  const int b = blockIdx.x;
  T* g = reinterpret_cast<T*>(a.gamma) + (int64_t)b * a.shot_elems;
  for (int s = threadIdx.x; s < S; s += blockDim.x) {
    const LocalDesc& d = locals0[s];
    for (int k = 0; k < d.P; ++k) g[d.off + k] = (k == 0) ? T(1) : T(0);
  }
  double* lam = a.lam + (int64_t)b * a.nbonds * a.chi;
  for (int w = threadIdx.x; w < a.nbonds * a.chi; w += blockDim.x) lam[w] = (w % a.chi == 0) ? 1.0 : 0.0;
  double* la = a.logacc + (int64_t)b * a.nslots;
  for (int w = threadIdx.x; w < a.nslots; w += blockDim.x) la[w] = 0.0;
}

// psi_s <- X^{m(s,t)} K psi_s on the physical leg, then divide by the power of two at or
// above the largest magnitude (an exact scaling; its log goes to the site's log-scale
// slot).  The mixing is computed in FP64 whatever the storage type: psi has entries of both
// signs, and a rounded FP32 sum would be an additive perturbation of the state.  One block
// per (site, shot); in place.
//
// What bounds it: FP64 instructions (19 cycles of an SM each), then memory.  Terms whose coefficient is
// zero (the vertical weights are diagonal) are left out -- exact zeros in sums that keep their order --,
// the largest magnitude is found on the upper words, of which only the exponent is used, the scaling
// is done in the exponent, and a thread keeps its mixed values where they fit: 2 FP64 instructions per
// pair of values instead of 16.  Measured: rotated d9 chi 8, 1000 shots 19.2 -> 14.8 ms of a decode.
//
// v 2^-e2 for a scaling that is exact (to a normal value): in the exponent, otherwise by multiplication.
__device__ __forceinline__ double local_scale(double v, int e2, double sc) {
  const unsigned hi = (unsigned)__double2hiint(v);
  const int ex = (int)((hi >> 20) & 0x7FFu);
  const int to = ex - e2;
  return ex > 0 && ex < 0x7FF && to > 0 && to < 0x7FF ? __hiloint2double((int)(hi - (unsigned)(e2 << 20)), __double2loint(v))
                                                     : v * sc;
}

template <typename T, int P>
__device__ __forceinline__ void local_site(const SweepArgs& a, const LocalDesc& d, const double* K, unsigned used, int b,
                                           int s, unsigned* red) {
  constexpr int KEEP = 16 / P;   // rows of a thread kept in registers (2 x 256 x KEEP values cover chi = 8)
  const T* g = reinterpret_cast<const T*>(a.gamma) + (int64_t)b * a.shot_elems + d.off;
  T* go = reinterpret_cast<T*>(a.gamma) + (int64_t)b * a.shot_elems + d.out_off;
  auto mix = [&](int r, double (&out)[P]) {
    double v[P];
#pragma unroll
    for (int k = 0; k < P; ++k) v[k] = double(g[(int64_t)k * d.rest + r]);
#pragma unroll
    for (int i = 0; i < P; ++i) {
      double acc = 0.0;
      bool first = true;   // the same for every thread
#pragma unroll
      for (int k = 0; k < P; ++k)
        if ((used >> (i * P + k)) & 1u) {
          acc = first ? K[i * P + k] * v[k] : acc + K[i * P + k] * v[k];
          first = false;
        }
      out[i] = acc;
    }
  };
  unsigned mx = 0u;   // the upper word of the largest magnitude
  auto top = [&](const double (&v)[P]) {
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const unsigned hi = (unsigned)__double2hiint(v[i]) & 0x7FFFFFFFu, lo = (unsigned)__double2loint(v[i]);
      mx = max(mx, hi | (unsigned)(hi == 0u && lo != 0u));   // a subnormal value counts by its presence
    }
  };
  double kept[KEEP][P];
#pragma unroll
  for (int u = 0; u < KEEP; ++u) {
    const int r = threadIdx.x + u * blockDim.x;
    if (r < d.rest) {
      mix(r, kept[u]);
      top(kept[u]);
    }
  }
  const int r1 = threadIdx.x + KEEP * blockDim.x;
  for (int r = r1; r < d.rest; r += blockDim.x) {
    double v[P];
    mix(r, v);
    top(v);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = 0u;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = max(mx, red[w]);
  int e2 = 0;
  const bool nz = mx > 0u;
  const bool over = mx >= 0x7FF00000u;   // infinity or NaN
  if (mx >= 0x00100000u && !over) e2 = (int)(mx >> 20) - 1022;   // normal: mx = f 2^e2, f in [1/2, 1)
  if (nz && mx < 0x00100000u) {
    // subnormal: as frexp of the value itself
    double m2 = 0.0;
    for (int r = threadIdx.x; r < d.rest; r += blockDim.x) {
      double v[P];
      mix(r, v);
#pragma unroll
      for (int i = 0; i < P; ++i) m2 = fmax(m2, fabs(v[i]));
    }
    __shared__ double red2[32];
    for (int o = 16; o > 0; o >>= 1) m2 = fmax(m2, __shfl_xor_sync(0xffffffffu, m2, o));
    if ((threadIdx.x & 31) == 0) red2[threadIdx.x >> 5] = m2;
    __syncthreads();
    m2 = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) m2 = fmax(m2, red2[w]);
    if (m2 > 0.0) frexp(m2, &e2);
  }
  const double sc = ldexp(1.0, -e2);        // exact
#pragma unroll
  for (int u = 0; u < KEEP; ++u) {
    const int r = threadIdx.x + u * blockDim.x;
    if (r < d.rest)
#pragma unroll
      for (int i = 0; i < P; ++i) go[(int64_t)i * d.rest + r] = T(local_scale(kept[u][i], e2, sc));
  }
  for (int r = r1; r < d.rest; r += blockDim.x) {
    double v[P];
    mix(r, v);
#pragma unroll
    for (int i = 0; i < P; ++i) go[(int64_t)i * d.rest + r] = T(local_scale(v[i], e2, sc));
  }
  if (threadIdx.x == 0) {
    double* la = a.logacc + (int64_t)b * a.nslots + s;
    *la += nz ? double(e2) * 0.69314718055994530942 : -INFINITY;
    if (over || non_finite(sc)) mark_non_finite(a, b);   // sc: no factor scales a value below 2^-1024 up
    if (a.rec_sc) a.rec_sc[(int64_t)b * gridDim.x + s] = sc;
  }
}

template <typename T>
__global__ void k_local(SweepArgs a, const LocalDesc* __restrict__ locals) {
  const int s = blockIdx.x, b = blockIdx.y;
  const LocalDesc& d = locals[s];
  __shared__ double K[kMaxPhys * kMaxPhys];
  __shared__ unsigned red[32];
  const int m = a.det[(int64_t)vshot_row(a.vs, a.wave_first, b) * a.n_det + d.det] & 1;
  const Override* o = vshot_ovr(a.vs, a.ovr, a.wave_first, b, kOvrLocal, a.layer * (int)gridDim.x + s);
  const double* Ksrc = o ? o->val : d.K;
  if (threadIdx.x < d.P * d.P) {
    const int row = threadIdx.x / d.P, col = threadIdx.x % d.P;
    K[threadIdx.x] = Ksrc[(row ^ m) * d.P + col];     // rows of X^m K
  }
  __syncthreads();
  unsigned used = 0u;   // coefficients that are not zero (tested on the bits: an FP64 comparison costs an FMA)
  for (int w = 0; w < d.P * d.P; ++w) used |= (unsigned)((__double_as_longlong(K[w]) << 1) != 0ll) << w;
  if (d.P == 2) local_site<T, 2>(a, d, K, used, b, s, red);
  else local_site<T, 4>(a, d, K, used, b, s, red);
}

// ---- launchers ---------------------------------------------------------------------------
template <typename T, typename R>
cudaError_t launch_sweep_init(const SweepArgs& a, const LocalDesc* locals0, int S, cudaStream_t st) {
  k_init<T><<<a.B, 256, 0, st>>>(a, locals0, S);
  return cudaGetLastError();
}

template <typename T, typename R>
cudaError_t launch_local(const SweepArgs& a, const LocalDesc* locals, int S, cudaStream_t st) {
  k_local<T><<<dim3(S, a.B), 256, 0, st>>>(a, locals);
  return cudaGetLastError();
}

template <typename T, typename R>
cudaError_t launch_round(const SweepArgs& a0, const GateDesc* gates, const Round& rd, double* gram, double* tbuf, int S,
                         cudaStream_t st, Prof* prof) {
  const GateDesc* g = gates + rd.first;
  const int D = std::max(rd.maxD, rd.maxDn);
  SweepArgs a = a0;
  const int cr = a0.chunk_rows > 0 ? a0.chunk_rows : kChunkRows;
  a.gram_chunks = absorb_chunks(rd.max_rows, cr);
  a.gate_base = rd.first;
  auto B = [&](int k) { if (prof) prof->begin(k); };
  auto E = [&](int k) { if (prof) prof->end(k); };
  B(TD_K_GRAM);
  cudaError_t e = (a.tc && gram_tc_supported(rd.maxD))
                      ? launch_gram_tc<T>(a, g, rd.count, rd.maxD, gram, a.gram_chunks, cr, st)
                      : launch_gram2<T>(a, g, rd.count, D, gram, a.gram_chunks, cr, st);
  E(TD_K_GRAM);
  if (e != cudaSuccess) return e;
  B(TD_K_CORE);
  e = launch_core2<R>(a, g, rd.count, rd.maxD, gram, tbuf, S, a.precond != 0, st);
  E(TD_K_CORE);
  if (e != cudaSuccess) return e;
  B(TD_K_UPDATE);
  e = launch_update2<T>(a, g, rd.count, D, tbuf, rd.max_rows, st);
  E(TD_K_UPDATE);
  return e;
}

template cudaError_t launch_sweep_init<double, double>(const SweepArgs&, const LocalDesc*, int, cudaStream_t);
template cudaError_t launch_sweep_init<float, float>(const SweepArgs&, const LocalDesc*, int, cudaStream_t);
template cudaError_t launch_local<double, double>(const SweepArgs&, const LocalDesc*, int, cudaStream_t);
template cudaError_t launch_local<float, float>(const SweepArgs&, const LocalDesc*, int, cudaStream_t);
template cudaError_t launch_round<double, double>(const SweepArgs&, const GateDesc*, const Round&, double*, double*,
                                                  int, cudaStream_t, Prof*);
template cudaError_t launch_round<float, float>(const SweepArgs&, const GateDesc*, const Round&, double*, double*, int,
                                                cudaStream_t, Prof*);

}  // namespace td
