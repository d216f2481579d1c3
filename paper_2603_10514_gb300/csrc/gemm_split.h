// gemm_split.h -- how the FP64 products (gemm_fp64.cu) are cut up: tiles of kGemmRows rows by bn
// columns, and the K steps of all tiles, in order, dealt to the CTAs in equal runs.
#pragma once

#include <algorithm>

#ifdef __CUDACC__
#define CHASE_HD __host__ __device__
#else
#define CHASE_HD
#endif

namespace chase {

constexpr int kGemmRows = 64, kGemmCols = 64;

struct GemmTile {
  int m0, n0, nb;   // first row and column, columns
  int t;            // number of the tile
  int kt;           // its K steps (tri: rows of B that are not zero)
  long long w0;     // K steps of the tiles before it
};

// `whole`: CTA g takes tile g.  Otherwise CTA g takes the K steps [begin(g), begin(g + 1)) of the
// sequence; a tile that is shared by CTAs g0 .. g1 has its parts in slots g + t, which no two parts
// share (from one part to the next g or t or both grow).
struct GemmSplit {
  int M, N, K, upper, tri;
  int bn, tn, tm, T, G, whole;
  long long W;

  CHASE_HD int rows_of(int n) const {  // row tiles of column tile n
    const int last = (N < (n + 1) * bn ? N : (n + 1) * bn) - 1;
    const int r = last / kGemmRows + 1;
    return upper && r < tm ? r : tm;
  }
  CHASE_HD int steps_of(int n) const {
    const int k = (n + 1) * bn;
    return tri && k < K ? k : K;
  }
  CHASE_HD GemmTile make(int n, int m, int t, long long w0) const {
    GemmTile g;
    g.m0 = m * kGemmRows;
    g.n0 = n * bn;
    g.nb = N - g.n0 < bn ? N - g.n0 : bn;
    g.t = t;
    g.kt = steps_of(n);
    g.w0 = w0;
    return g;
  }
  CHASE_HD GemmTile tile(int t) const {
    int n = 0, t0 = 0;
    long long w = 0;
    while (n + 1 < tn && t - t0 >= rows_of(n)) {
      t0 += rows_of(n);
      w += (long long)rows_of(n) * steps_of(n);
      ++n;
    }
    return make(n, t - t0, t, w + (long long)(t - t0) * steps_of(n));
  }
  CHASE_HD GemmTile at(long long w) const {  // the tile of K step w < W
    int n = 0, t0 = 0;
    long long b = 0;
    while (n + 1 < tn && w - b >= (long long)rows_of(n) * steps_of(n)) {
      t0 += rows_of(n);
      b += (long long)rows_of(n) * steps_of(n);
      ++n;
    }
    const int m = (int)((w - b) / steps_of(n));
    return make(n, m, t0 + m, b + (long long)m * steps_of(n));
  }
  CHASE_HD long long begin(int g) const { return (long long)g * W / G; }
  CHASE_HD int owner(long long w) const { return (int)(((w + 1) * G - 1) / W); }
  CHASE_HD long long slots() const { return whole ? 0 : (long long)G + T; }
  CHASE_HD long long slot_elems() const { return (long long)kGemmRows * bn; }
};

// kmin: fewest K steps a CTA is started for; room: elements of scratch memory for the parts.
inline GemmSplit gemm_split(int M, int N, int K, bool upper, bool tri, int ctas, int kmin, long long room) {
  GemmSplit s{};
  s.M = M;
  s.N = N;
  s.K = K > 0 ? K : 0;
  s.upper = upper;
  s.tri = tri;
  s.tn = (N + kGemmCols - 1) / kGemmCols;
  s.bn = (N + s.tn - 1) / s.tn;
  s.tn = (N + s.bn - 1) / s.bn;
  s.tm = (M + kGemmRows - 1) / kGemmRows;
  for (int n = 0; n < s.tn; ++n) {
    s.T += s.rows_of(n);
    s.W += (long long)s.rows_of(n) * s.steps_of(n);
  }
  s.G = (int)std::min<long long>(ctas, s.W / kmin);
  s.whole = s.G < 1 || (s.G < ctas && s.G <= s.T) || s.slots() * s.slot_elems() > room;
  if (s.whole) s.G = s.T;
  return s;
}

}  // namespace chase
