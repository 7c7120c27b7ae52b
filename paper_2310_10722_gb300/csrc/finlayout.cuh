// Leading dimensions and region sizes of the final contraction's matrices (final.cu, api.cu): usable on the host
// too, where the tests check the one against the other.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define TD_LAYOUT_HD __host__ __device__ __forceinline__
#else
#define TD_LAYOUT_HD inline
#endif

namespace td {

// Lanes per column pair used by team_svd_onesided for a team of nt threads and an m x n
// matrix, and a leading dimension for 4-byte elements that puts the g-lane windows of
// consecutive columns on disjoint shared-memory banks (ld = g mod 32).
TD_LAYOUT_HD int team_svd_group(int nt, int m, int n) {
  const int half = (n + (n & 1)) / 2;
  int g = half > 0 ? nt / half : 32;
  if (g < 1) g = 1;
  if (g > 32) g = 32;
  int p2 = 1;
  while (2 * p2 <= g) p2 *= 2;
  g = p2;
  const int rows_max = m > n ? m : n;
  while (g > 1 && g > rows_max) g >>= 1;
  return g;
}
TD_LAYOUT_HD int bank_ld32(int rows, int g) { return (rows + 31) / 32 * 32 + (g & 31); }

// The regions of M^T (n x m, n <= n_max, m <= m_max) and of the rotation V (m x m): their size at the widest
// cuts.  A smaller cut may have other lane groups and with them a larger leading dimension.
inline int64_t final_mt_elems(int nt, int n_max, int m_max) {
  int64_t e = 0;
  for (int m = 1; m <= m_max; ++m) {
    const int64_t x = (int64_t)m * bank_ld32(n_max, team_svd_group(nt, n_max, m));
    e = x > e ? x : e;
  }
  return e;
}
inline int64_t final_v_elems(int nt, int n_max, int m_max) {
  int64_t e = 0;
  for (int m = 1; m <= m_max; ++m) {
    const int64_t x = (int64_t)m * bank_ld32(m, team_svd_group(nt, n_max, m));
    e = x > e ? x : e;
  }
  return e;
}

// Leading dimension of `cols` columns of `rows` elements for groups of g lanes in a region of `room` elements:
// bank_ld32, or the unspread one where that does not fit (which always does: rows and cols are at most the
// widest cut's).  Without this, cuts of up to 31 rows ran past their region at small caps: in blocks of 256
// threads at chi_mps x bond = 16 and at chi_mps = 1 with bonds 8 to 11, in larger ones at up to 31.
TD_LAYOUT_HD int final_ld(int rows, int g, int cols, int64_t room) {
  const int ld = bank_ld32(rows, g);
  return (int64_t)cols * ld <= room ? ld : bank_ld32(rows, 0);
}

}  // namespace td
