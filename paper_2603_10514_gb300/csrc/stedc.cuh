// stedc.cuh -- the steps of one merge of the divide-and-conquer eigensolver for real
// symmetric tridiagonal matrices (Cuppen's rank-one tearing; Gu & Eisenstat, "A
// divide-and-conquer algorithm for the symmetric tridiagonal eigenproblem", 1995): deflation,
// the secular equation's roots (Li's middle way inside a bracket), and the vector z that makes
// the computed roots exact, so that the eigenvectors are orthogonal to working precision.
//
// Every step is written for a group of threads G (tid, size, sync, max over the group) or for
// `width` lanes L of a warp (sums and products over them, any over the whole warp); eigh.cu runs
// them over a warp, a CTA or a grid.  The groups of one warp call the L steps together: one that
// has no item of its own takes another's and writes nothing (write = false).  All loops are
// bounded, and every index written is below m whatever the data (NaN included).
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define DC_FN __device__ __forceinline__
#else
#define DC_FN inline
#endif

namespace chase {
namespace dc {

constexpr double kEps = 1.1102230246251565e-16;  // 2^-53

// k with 2^k x in [0.5, 1) (0 for 0, infinity and NaN).  The steps below square and invert what they
// are given, so a tridiagonal is first multiplied by 2^k of its largest entry, which rounds nothing.
DC_FN int scale_of(double x) {
  if (!(x > 0.0) || x - x != 0.0) return 0;
  int e;
  frexp(x, &e);
  return -e;
}

// One merge: the eigensystems of two adjacent tridiagonal blocks (n1 and m - n1 rows) and the
// coupling rho between them.  All arrays hold m entries.
struct Merge {
  int m, n1;
  double rho;         // 2 |e| of the torn off-diagonal (z is scaled by 1 / sqrt 2)
  double sign;        // its sign
  const double* D;    // eigenvalues, ascending within each half
  double *ds, *zs;    // sorted eigenvalues and z
  int* perm;          // sorted position -> column of Q
  unsigned char *small, *close, *type;
  int* idx;           // the K positions that remain, ascending
  int* defl;          // the m - K that deflate
  double *dl, *w;     // poles and weights of the secular equation
  int* pos;           // pole -> row of U (columns of Q that live in the first half first)
  int* gat;           // row of U -> column of Q
  double *mu, *zh;    // roots relative to pole org, corrected z
  int* org;
  double* lam;
  int *rp, *rq;       // rotations of Q's columns by deflated pairs, in order
  double *rc, *rs;
  int* dest;          // new position of root k (k < K) and of defl[t] (at K + t)
  int* cnt;           // K, rows of U from the first half alone, those or mixed, rotations
};

// z, the sorted order and the deflation of one merge; q_last / q_first: row n1 - 1 of the first
// and row n1 of the second block's eigenvectors (stride ldq).
template <class G>
DC_FN void setup(const G& g, const Merge& M, const double* q_last, const double* q_first, int ldq) {
  const int m = M.m, n1 = M.n1, n2 = m - n1;
  const double rsq2 = 0.70710678118654752440;
  for (int i = g.tid; i < m; i += g.size) M.perm[i] = i;
  g.sync();
  for (int i = g.tid; i < m; i += g.size) {
    const double d = M.D[i];
    // position of D[i] in the merged order (equal values: the first half's first)
    int lo = 0, hi = i < n1 ? n2 : n1;
    const double* other = i < n1 ? M.D + n1 : M.D;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      const bool before = i < n1 ? other[mid] < d : other[mid] <= d;
      if (before) lo = mid + 1; else hi = mid;
    }
    const int r = lo + (i < n1 ? i : i - n1);
    const double z = i < n1 ? q_last[(size_t)i * ldq] : M.sign * q_first[(size_t)(i - n1) * ldq];
    M.perm[r] = i;
    M.ds[r] = d;
    M.zs[r] = z * rsq2;
    M.type[i] = i < n1 ? 0 : 2;
  }
  g.sync();
  double zm = 0.0;
  for (int i = g.tid; i < m; i += g.size) zm = fmax(zm, fabs(M.zs[i]));
  zm = g.max(zm);
  const double dm = fmax(fabs(M.ds[0]), fabs(M.ds[m - 1]));
  // relative to D + rho z z^T (the eigenvalues carry the matrix's scale, z is a unit vector)
  const double tol = 8.0 * kEps * fmax(dm, M.rho * zm);
  for (int r = g.tid; r < m; r += g.size) {
    const double z = M.zs[r];
    M.small[r] = !(M.rho * fabs(z) > tol);
    unsigned char c = 0;
    if (r > 0) {
      const double y = M.zs[r - 1];
      c = !(fabs((M.ds[r] - M.ds[r - 1]) * z * y) > tol * (z * z + y * y));
    }
    M.close[r] = c;
  }
  g.sync();
  if (g.tid == 0) {
    int K = 0, nd = 0, nr = 0, pj = -1;
    bool moved = false;  // pj's z and d were changed by a rotation
    for (int r = 0; r < m; ++r) {
      if (M.small[r]) { M.defl[nd++] = r; continue; }
      if (pj < 0) { pj = r; moved = false; continue; }
      bool cl = M.close[r];
      if (moved || pj != r - 1) {
        const double z = M.zs[r], y = M.zs[pj];
        cl = !(fabs((M.ds[r] - M.ds[pj]) * z * y) > tol * (z * z + y * y));
      }
      if (cl) {  // rotate z[pj] into z[r]; the pair's coupling is below tol
        const double z = M.zs[r], y = M.zs[pj], t = sqrt(z * z + y * y);
        const double c = z / t, s = -y / t;
        const double dp = M.ds[pj], dr = M.ds[r];
        M.zs[r] = t;
        M.zs[pj] = 0.0;
        M.ds[pj] = dp * c * c + dr * s * s;
        M.ds[r] = dp * s * s + dr * c * c;
        const int p = M.perm[pj], q = M.perm[r];
        M.rp[nr] = p; M.rq[nr] = q; M.rc[nr] = c; M.rs[nr] = s;
        ++nr;
        if (M.type[p] != M.type[q]) M.type[p] = M.type[q] = 1;
        M.defl[nd++] = pj;
        moved = true;
      } else {
        M.idx[K++] = pj;
        moved = false;
      }
      pj = r;
    }
    if (pj >= 0) M.idx[K++] = pj;
    // rows of U: columns of the first half alone, mixed ones, columns of the second alone
    int c0 = 0, c1 = 0;
    for (int k = 0; k < K; ++k) {
      const int t = M.type[M.perm[M.idx[k]]];
      c0 += t == 0;
      c1 += t == 1;
    }
    int at[3] = {0, c0, c0 + c1};
    for (int k = 0; k < K; ++k) {
      const int col = M.perm[M.idx[k]];
      const int p = at[M.type[col]]++;
      M.pos[k] = p;
      M.gat[p] = col;
    }
    M.cnt[0] = K;
    M.cnt[1] = c0;
    M.cnt[2] = c0 + c1;
    M.cnt[3] = nr;
  }
  g.sync();
  const int K = M.cnt[0];
  for (int k = g.tid; k < K; k += g.size) {
    M.dl[k] = M.ds[M.idx[k]];
    M.w[k] = M.zs[M.idx[k]];
  }
  g.sync();
}

// Root k of 1 / rho + sum_i w_i^2 / (d_i - x) = 0 as mu = x - d_org, d_org the nearer pole.
template <class L>
DC_FN void root(const L& l, int K, int k, bool write, const double* dl, const double* w, double rho,
                double* mu_out, int* org_out, double* lam_out) {
  if (K == 1) {
    if (l.lane == 0 && write) { *mu_out = rho * w[0] * w[0]; *org_out = 0; *lam_out = dl[0] + rho * w[0] * w[0]; }
    return;
  }
  const double ri = 1.0 / rho;
  const bool inner = k < K - 1;
  const int a = inner ? k : K - 2, b = a + 1;  // the two poles of the interpolation
  const double gap = dl[b] - dl[a], h = 0.5 * gap;
  // inner: the other terms of f in the middle of the interval; last: |w|^2
  double s = 0.0;
  for (int i = l.lane; i < K; i += l.width) {
    const double t = inner ? w[i] / ((dl[i] - dl[a]) - h) : w[i];
    if (!inner || (i != a && i != b)) s += w[i] * t;
  }
  s = l.sum(s);
  int org = b;
  double lo = 0.0, hi, mu;
  if (inner) {
    const double c = ri + s, wa = w[a] * w[a], wb = w[b] * w[b];
    const bool left = c + (wb - wa) / h > 0.0;  // f(middle) > 0: the root lies in the left half
    const double A = left ? c * gap + wa + wb : c * gap - wa - wb, B = left ? wa * gap : wb * gap;
    const double q = sqrt(fabs(A * A + (left ? -4.0 : 4.0) * B * c));
    if (left) {
      org = a;
      hi = h;
      mu = A > 0.0 ? 2.0 * B / (A + q) : (A - q) / (2.0 * c);
    } else {
      lo = -h;
      hi = 0.0;
      mu = A < 0.0 ? 2.0 * B / (A - q) : -(A + q) / (2.0 * c);
    }
  } else {
    hi = rho * s * (1.0 + 4.0 * kEps);
    mu = 0.5 * hi;
  }
  if (!(mu > lo && mu < hi)) mu = 0.5 * (lo + hi);
  const double dorg = dl[org];
  bool act = true;
  for (int it = 0; it < 80; ++it) {
    double psi = 0.0, phi = 0.0, dpsi = 0.0, dphi = 0.0;
    for (int i = l.lane; i < K; i += l.width) {
      const double t = w[i] / ((dl[i] - dorg) - mu);
      if (i <= a) { psi += w[i] * t; dpsi += t * t; }
      else { phi += w[i] * t; dphi += t * t; }
    }
    psi = l.sum(psi); phi = l.sum(phi); dpsi = l.sum(dpsi); dphi = l.sum(dphi);
    const double f = ri + psi + phi, df = dpsi + dphi;
    act = act && fabs(f) > kEps * (8.0 * (fabs(psi) + fabs(phi)) + ri + fabs(mu) * df);
    if (!l.any(act)) break;
    if (act) {
      if (f > 0.0) hi = mu; else lo = mu;
      const double Da = (dl[a] - dorg) - mu, Db = (dl[b] - dorg) - mu;
      double c = f - Da * dpsi - Db * dphi;
      const double A = (Da + Db) * f - Da * Db * df, B = Da * Db * f;
      // the middle way's step: inner roots (A - q) / 2c, the last one (A + q) / 2|c|
      double sg = 1.0;
      if (inner) sg = -1.0;
      else c = fabs(c);
      const double q = sqrt(fabs(A * A - 4.0 * B * c));
      const bool direct = inner ? A <= 0.0 : A >= 0.0;
      const double num = direct ? A + sg * q : 2.0 * B, den = direct ? 2.0 * c : A - sg * q;
      double eta = num / den;
      if (c == 0.0) eta = inner ? B / A : hi - mu;
      if (!(f * eta < 0.0)) eta = -f / df;
      double nx = mu + eta;
      if (!(nx > lo && nx < hi)) nx = 0.5 * (lo + hi);
      if (nx == mu || !(nx > lo && nx < hi)) act = false;  // the bracket is down to neighbours
      else mu = nx;
    }
  }
  if (l.lane == 0 && write) { *mu_out = mu; *org_out = org; *lam_out = dorg + mu; }
}

// z_i for which the computed roots are the exact ones (Loewner's formula).
template <class L>
DC_FN void zhat(const L& l, int K, int i, bool write, const double* dl, const double* w, const double* mu,
                const int* org, double* zh) {
  const double di = dl[i];
  double p = 1.0;
  for (int j = l.lane; j < K; j += l.width) {
    const double t = (di - dl[org[j]]) - mu[j];
    p *= (j == i) ? t : t / (di - dl[j]);
  }
  p = l.prod(p);
  if (l.lane == 0 && write) zh[i] = copysign(sqrt(fabs(p)), w[i]);
}

// Column j of U (eigenvector of the rank-one update), rows in gather order, unit length.
template <class L>
DC_FN void ucol(const L& l, int K, int j, bool write, const double* dl, const double* zh, const double* mu,
                const int* org, const int* pos, double* U, int ldu) {
  const double dorg = dl[org[j]], m = mu[j];
  double s = 0.0;
  for (int i = l.lane; i < K; i += l.width) {
    const double u = zh[i] / ((dl[i] - dorg) - m);
    s += u * u;
  }
  const double r = 1.0 / sqrt(l.sum(s));
  if (write)
    for (int i = l.lane; i < K; i += l.width) U[(size_t)pos[i] + (size_t)j * ldu] = zh[i] / ((dl[i] - dorg) - m) * r;
}

// New position of value t (t < K: root t; else the deflated value t - K).  One count for both kinds:
// the groups of a warp may hold both, and its lanes have to meet in the same shuffles.
template <class L>
DC_FN void place(const L& l, const Merge& M, int K, int t, bool write) {
  const int nd = M.m - K;
  const bool is_root = t < K;
  const double v = is_root ? M.lam[t] : M.ds[M.defl[t - K]];
  int n = 0;
  if (is_root) {
    for (int u = l.lane; u < nd; u += l.width) n += M.ds[M.defl[u]] < v;
  } else {
    const int me = t - K;
    for (int k = l.lane; k < K; k += l.width) n += M.lam[k] <= v;
    for (int u = l.lane; u < nd; u += l.width) {
      const double x = M.ds[M.defl[u]];
      n += x < v || (x == v && u < me);
    }
  }
  n = l.count(n) + (is_root ? t : 0);
  if (l.lane == 0 && write) M.dest[t] = n;
}

}  // namespace dc
}  // namespace chase
