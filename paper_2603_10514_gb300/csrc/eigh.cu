// eigh.cu -- direct eigensolver of the Rayleigh-Ritz step (Algorithm 1: solve A~ W = W Lambda~)
// and of the Lanczos runs' tridiagonals.
//
//   1. Householder reduction of the Hermitian H (l x l) to a real tridiagonal T = Q^H H Q, one
//      cooperative kernel: columns are dealt to the CTAs in turn and stay in shared memory.
//      Per column every CTA forms its entries of H v from its own columns (H is Hermitian, so
//      no partial sums cross CTAs); after the step's one grid barrier every CTA forms
//      w itself, the owner's next raw column was published beside it, and the next reflector
//      is formed by every CTA from that while its other warps apply H -= v w^H + w v^H.
//   2. Divide and conquer for T = Z Lambda Z^T (stedc.cuh): blocks of up to 32 rows in one CTA
//      each, then per level five launches over all merges of the level.
//   3. W = Q Z: one warp per column of W applies the reflectors, eight at a time; columns are
//      independent, so no CTA waits for another.
// It replaces a cyclic Jacobi iteration.  GB300 issues 2 FP64 FMAs per clock per SM, which binds
// both: Jacobi takes ~5 sweeps of ~9 l^3 (complex: x 4) FMAs and l - 1 grid-wide rounds each,
// this ~4 l^3 for step 1, ~l^3 (real) for 2 and ~2 l^3 for 3, and l grid barriers in all.
// Measured (random H, GB300): l = 600 complex 124 -> 10.3 ms (6.4 reduction, 1.75 divide and
// conquer, 2.05 back-transformation), l = 230 complex 31 -> 3.0, l = 600 real 80 -> 6.7, l = 30
// real 2.0 -> 0.41.
//
// H and then T are multiplied by powers of two that bring their largest entries to [0.5, 1), the
// eigenvalues back at the end, so squares and reciprocals stay in range at every scale.
// Every wait is bounded; a CTA that waits too long raises an abort flag that the others see, and
// the kernel sets DevStatus.timeout.  Sums are taken in fixed orders: results are reproducible.
// A non-finite T gives NaN eigenvalues and vectors.
#include "../../include/chase_gb300.h"
#include "common.cuh"
#include "kernels.h"
#include "stedc.cuh"

#include <type_traits>

#define TRY_EIG(x)           \
  do {                       \
    int _rc = (x);           \
    if (_rc) return _rc;     \
  } while (0)

namespace chase {

namespace {

constexpr int TNT = 256;          // threads of the reduction kernel
constexpr int LEAF = 32;          // rows of a divide-and-conquer leaf
constexpr size_t kSmemMax = 227 * 1024;

__device__ __forceinline__ double warp_add(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_addt(double v) { return warp_add(v); }
__device__ __forceinline__ z64 warp_addt(z64 v) { return z64{warp_add(v.x), warp_add(v.y)}; }

template <class T> __device__ __forceinline__ T ld_cg(const T* p);
template <> __device__ __forceinline__ double ld_cg<double>(const double* p) { return __ldcg(p); }
template <> __device__ __forceinline__ z64 ld_cg<z64>(const z64* p) {
  const double2 v = __ldcg((const double2*)p);
  return z64{v.x, v.y};
}

__device__ __forceinline__ double im_of(double) { return 0.0; }
__device__ __forceinline__ double im_of(z64 a) { return a.y; }

// ---------------------------------------------------------------------------
// 1. Reduction to tridiagonal form
// ---------------------------------------------------------------------------
// H (l x l, ld ldh): column j is overwritten by reflector j (rows j + 1 ..).  in_smem: this CTA's
// columns are kept in shared memory, else in place.  Per column j, with v = v_j and tau known to
// every CTA:
//   x_c = tau (H v)_c for the own columns c; the owner of column j + 1 publishes it as it is;
//   grid barrier; alpha = -1/2 tau x^H v (real: -1/2 |tau|^2 v^H H v) from the CTAs' parts;
//   every CTA updates column j + 1 for itself and forms reflector j + 1 from it -- a few l FMAs
//   more on every SM, but no second wait on its owner -- and while one warp takes the reflector's
//   square root and divisions (~35 dependent FP64 instructions), the others apply
//   H -= v w^H + w v^H, w = x + alpha v, to the own columns.
// All of it on 2^ex H, with its largest entry in [0.5, 1): the squares of the norms stay in range.
// xb, cb: 2 l elements, part: 2 G doubles; scr: 3 l elements per CTA where they do not fit
// shared memory (else null); ex: one int, written.
template <class T>
__global__ void __launch_bounds__(TNT) tridiag_kernel(int l, T* H, int ldh, int in_smem, T* tau, double* d,
                                                      double* e, T* xb, T* cb, double* part, T* scr, int* ex,
                                                      GridBar* gb, DevStatus* dst) {
  extern __shared__ __align__(16) unsigned char tri_smem[];
  const int G = gridDim.x, me = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = TNT / 32;
  __shared__ double sh[NW];
  __shared__ T sh_tau, sh_scale;
  __shared__ double sh_alpha;
  __shared__ long long sh_max[NW];
  const int own = (l + G - 1) / G;                     // columns me, me + G, ...
  const int nc = me < l ? (l - 1 - me) / G + 1 : 0;
  T* sp = (T*)tri_smem;                                // 4 partial sums per own column
  T* sq = sp + 4 * own;                                // the update's two factors per own column
  T* vec = scr ? scr + (size_t)me * 3 * l : sq + 2 * own;
  T *vs = vec, *xs = vec + l, *us = vec + 2 * (size_t)l;
  T* S = scr ? sq + 2 * own : vec + 3 * (size_t)l;
  auto column = [&](int k) -> T* { return in_smem ? S + (size_t)k * l : H + (size_t)(me + k * G) * ldh; };
  long long mx = 0;  // bits of the largest |re|, |im| of the own columns
  auto bits = [](double x) { return __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll; };
  for (int k = 0; k < nc; ++k)
    for (int i = tid; i < l; i += TNT) {
      const T h = H[(size_t)i + (size_t)(me + k * G) * ldh];
      if (in_smem) S[(size_t)k * l + i] = h;
      mx = max(mx, max(bits(Sc<T>::re(h)), bits(im_of(h))));
    }
  auto block_maxbits = [&](long long v) {
    for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) sh_max[warp] = v;
    __syncthreads();
    for (int w = 0; w < NW; ++w) v = max(v, sh_max[w]);
    return v;
  };
  mx = block_maxbits(mx);

  // Reflector j from u (rows j .. of the updated column j): its scalars, by one thread.
  auto scalars = [&](int j, const T* u) {
    double x2 = 0.0;
    for (int w = 0; w < NW; ++w) x2 += sh[w];
    const T alpha = u[j + 1];
    const double ar = Sc<T>::re(alpha), ai = im_of(alpha);
    T t = Sc<T>::zero(), sc = Sc<T>::zero();
    double beta = ar;
    const double nn = ar * ar + ai * ai + x2;
    if ((x2 != 0.0 || ai != 0.0) && !(nn < 1e-300)) {  // (below: nothing is left of a matrix of norm 1, and 1 / nn overflows)
      const double rn = rsqrt(nn);
      beta = -copysign(nn * rn, ar);
      const double ib = -copysign(rn, ar), dr = ar - beta, id = 1.0 / (dr * dr + ai * ai);
      if constexpr (Sc<T>::cplx) {
        t = z64{(beta - ar) * ib, -ai * ib};
        sc = z64{dr * id, -ai * id};
      } else {
        t = (beta - ar) * ib;
        sc = dr * id;
      }
    }
    sh_tau = t;
    sh_scale = sc;
    if (j % G == me) {
      d[j] = Sc<T>::re(u[j]);
      e[j] = beta;
      tau[j] = t;
    }
  };
  auto norm_part = [&](double s) {  // sum of squares below the subdiagonal, a part per warp
    s = warp_add(s);
    if (lane == 0) sh[warp] = s;
  };
  // v = u scaled (in u's place), kept in H by its owner
  auto finish_reflector = [&](int j, T* u) {
    const T sc = sh_scale;
    T* hcol = H + (size_t)j * ldh;
    for (int i = j + 1 + tid; i < l; i += TNT) {
      const T v = (i == j + 1) ? Sc<T>::one() : Sc<T>::mul(u[i], sc);
      u[i] = v;
      if (j % G == me) hcol[i] = v;
    }
  };

  // reflector 0, by every CTA from the matrix (read before any column is overwritten: its owner
  // writes it after the first barrier's worth of work is published, see below)
  for (int i = tid; i < l; i += TNT) us[i] = H[i];
  unsigned bars = 0;
  int par = 0;
  if (G > 1) {
    if (tid == 0) ((long long*)part)[me] = mx;
    if (!grid_barrier(gb, G, bars)) {  // column 0 has been read everywhere
      if (tid == 0) atomicOr(&dst->timeout, 16);
      return;
    }
    for (int b = tid; b < G; b += TNT) mx = max(mx, __ldcg((const long long*)part + b));
    mx = block_maxbits(mx);
    par = 1;  // the first step writes the other half of `part`: this one may still be read
  }
  const int sx = dc::scale_of(__longlong_as_double(mx));
  if (me == 0 && tid == 0) *ex = sx;
  // (two factors: 2^sx alone may be out of range)
  const double f0 = ldexp(1.0, sx / 2), f1 = ldexp(1.0, sx - sx / 2);
  auto scaled = [&](T h) { return Sc<T>::scale(Sc<T>::scale(h, f0), f1); };
  if (sx != 0)
    for (int k = 0; k < nc; ++k)
      for (int i = tid; i < l; i += TNT) column(k)[i] = scaled(column(k)[i]);
  {
    double s = 0.0;
    for (int i = tid; i < l; i += TNT) {
      const T h = scaled(us[i]);
      us[i] = h;
      if (i >= 2) s += Sc<T>::abs2(h);
    }
    norm_part(s);
  }
  __syncthreads();
  if (l == 1) {
    if (me == 0 && tid == 0) d[0] = Sc<T>::re(us[0]);
    return;
  }
  if (tid == 0) scalars(0, us);
  __syncthreads();
  finish_reflector(0, us);
  __syncthreads();
  for (int j = 0; j + 1 < l; ++j) {
    { T* q = vs; vs = us; us = q; }  // v_j
    const T t = sh_tau;
    const int k0 = (j + 1 <= me) ? 0 : (j + 1 - me + G - 1) / G, na = nc - k0;  // own columns >= j + 1
    const bool trivial = Sc<T>::re(t) == 0.0 && im_of(t) == 0.0;
    T *xg = xb + (size_t)par * l, *cg = cb + (size_t)par * l;
    const bool next_mine = (j + 1) % G == me;
    // x = tau H v on the own columns, each split over enough warps to use every sub-partition
    if (!trivial) {
      const int parts = na <= 2 ? 4 : na <= 4 ? 2 : 1;
      for (int w = warp; w < na * parts; w += NW) {
        const int k = k0 + w / parts, p = w - (k - k0) * parts;
        const T* col = column(k);
        T s = Sc<T>::zero();
        for (int i = j + 1 + 32 * p + lane; i < l; i += 32 * parts) Sc<T>::fmac(s, col[i], vs[i]);
        s = warp_addt(s);
        if (lane == 0) sp[(size_t)k * 4 + p] = s;
      }
      __syncthreads();
      if (warp == 0) {
        double a = 0.0;
        for (int k = k0 + lane; k < nc; k += 32) {
          T s = sp[(size_t)k * 4];
          for (int p = 1; p < parts; ++p) s = Sc<T>::add(s, sp[(size_t)k * 4 + p]);
          s = Sc<T>::mul(t, s);
          const int c = me + k * G;
          if (G > 1) xg[c] = s;
          else xs[c] = s;
          a += Sc<T>::re(Sc<T>::mul(t, Sc<T>::mul(Sc<T>::conj(s), vs[c])));
        }
        if (na <= 1) a = __shfl_sync(0xffffffffu, a, 0);
        else a = warp_add(a);
        if (lane == 0) {
          if (G > 1) part[(size_t)par * G + me] = a;
          else sh_alpha = -0.5 * a;
        }
      }
    }
    if (G > 1) {
      if (next_mine)
        for (int i = j + 1 + tid; i < l; i += TNT) cg[i] = column(k0)[i];
      if (!grid_barrier(gb, G, bars)) {
        if (tid == 0) atomicOr(&dst->timeout, 16);
        return;
      }
      if (warp == 0) {
        if (!trivial) {
          double a = 0.0;
          for (int b = lane; b < G; b += 32) a += __ldcg(part + (size_t)par * G + b);
          a = warp_add(a);
          if (lane == 0) sh_alpha = -0.5 * a;
        }
      } else {
        for (int i = j + 1 + tid - 32; i < l; i += TNT - 32) {
          if (!trivial) xs[i] = ld_cg(xg + i);
          us[i] = ld_cg(cg + i);
        }
      }
      par ^= 1;
    } else {
      __syncthreads();
      for (int i = j + 1 + tid; i < l; i += TNT) us[i] = column(k0)[i];
    }
    __syncthreads();
    const double al = trivial ? 0.0 : sh_alpha;
    // H[:, c] -= v conj(w_c) + w conj(v_c) = v q + x p with q = -(conj(x_c) + 2 alpha conj(v_c)),
    // p = -conj(v_c)
    auto factors = [&](int c, T* q, T* p) {
      const T vc = Sc<T>::conj(vs[c]);
      *q = Sc<T>::scale(Sc<T>::add(Sc<T>::conj(xs[c]), Sc<T>::scale(vc, 2.0 * al)), -1.0);
      *p = Sc<T>::scale(vc, -1.0);
    };
    if (!trivial) {
      T q, p;
      factors(j + 1, &q, &p);
      double s = 0.0;
      for (int i = j + 1 + tid; i < l; i += TNT) {
        T h = us[i];
        Sc<T>::fma(h, vs[i], q);
        Sc<T>::fma(h, xs[i], p);
        us[i] = h;
        if (i >= j + 3) s += Sc<T>::abs2(h);
      }
      norm_part(s);
      for (int k = k0 + tid; k < nc; k += TNT) factors(me + k * G, sq + 2 * k, sq + 2 * k + 1);
    } else {
      double s = 0.0;
      for (int i = j + 3 + tid; i < l; i += TNT) s += Sc<T>::abs2(us[i]);
      norm_part(s);
    }
    __syncthreads();
    if (j + 2 == l) {  // the last diagonal entry
      if (next_mine && tid == 0) d[j + 1] = Sc<T>::re(us[j + 1]);
      return;
    }
    if (tid == 0) scalars(j + 1, us);
    if (!trivial && warp != 0 && warp != NW / 2) {  // (warp NW / 2 shares warp 0's FP64 pipe)
      // chunks of 32 rows of every own column after j + 1, over the other warps
      const int wi = warp < NW / 2 ? warp - 1 : warp - 2, kf = k0 + (next_mine ? 1 : 0);
      const int ch = (l - j - 1 + 31) / 32;
      for (int w = wi; w < (nc - kf) * ch; w += NW - 2) {
        const int k = kf + w / ch, i = j + 1 + 32 * (w - (k - kf) * ch) + lane;
        if (i < l) {
          T* col = column(k);
          T h = col[i];
          Sc<T>::fma(h, vs[i], sq[2 * k]);
          Sc<T>::fma(h, xs[i], sq[2 * k + 1]);
          col[i] = h;
        }
      }
    }
    __syncthreads();
    finish_reflector(j + 1, us);
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// 2. Divide and conquer
// ---------------------------------------------------------------------------
struct CtaGroup {
  int tid, size;
  double* red;
  __device__ void sync() const { __syncthreads(); }
  __device__ double max(double v) const {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if ((tid & 31) == 0) red[tid >> 5] = v;
    __syncthreads();
    for (int w = 0; w < (size >> 5); ++w) v = fmax(v, red[w]);
    return v;
  }
};
// `size` threads of a CTA (whole warps, in a row) with a barrier of their own.
struct PartGroup {
  int tid, size, id;
  double* red;
  __device__ void sync() const { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(size) : "memory"); }
  __device__ double max(double v) const {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    sync();
    if ((tid & 31) == 0) red[tid >> 5] = v;
    sync();
    for (int w = 0; w < (size >> 5); ++w) v = fmax(v, red[w]);
    return v;
  }
};
struct WarpGroup {
  int tid, size;
  __device__ void sync() const { __syncwarp(); }
  __device__ double max(double v) const {
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
  }
};
// `width` lanes (a power of two) of a warp, `group` of them counted.
struct Lanes {
  int lane, width, group;
  __device__ explicit Lanes(int w) : lane(threadIdx.x & (w - 1)), width(w), group((threadIdx.x & 31) / w) {}
  __device__ double sum(double v) const {
    for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
  __device__ double prod(double v) const {
    for (int o = width >> 1; o > 0; o >>= 1) v *= __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
  __device__ int count(int v) const {
    for (int o = width >> 1; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
  }
  __device__ bool any(bool v) const { return __any_sync(0xffffffffu, v); }
};
// f(i, write) for the items [0, n) of a merge, one per group of lanes: warp w of nw.
template <class F>
__device__ __forceinline__ void for_items(const Lanes& L, int w, int nw, int n, const F& f) {
  const int per = 32 / L.width;
  for (int i0 = w * per; i0 < n; i0 += nw * per) {
    const int i = i0 + L.group;
    f(min(i, n - 1), i < n);
  }
}

// Arrays of one problem of order n (offsets of `batch` problems are uniform strides).
struct DcWork {
  int n;
  double* D[2];
  double *ds, *zs, *dl, *w, *mu, *zh, *lam, *rc, *rs;
  double* es;        // off-diagonal entries of 2^ex T
  int *perm, *idx, *defl, *pos, *gat, *org, *rp, *rq, *dest, *cnt;
  unsigned char *small, *close, *type;
  double *Q[2], *U;  // n x n
  int* bad;          // T was not finite
  int* ex;           // D holds the eigenvalues of 2^ex T (see dc::scale_of)
};
constexpr int kDcDoubles = 12, kDcInts = 13, kDcBytes = 3;

__host__ __device__ inline size_t dc_align(size_t x) { return (x + 255) & ~(size_t)255; }
// mats: n x n matrices among them (Q[0], or with Q[1] and U).
inline size_t dc_bytes(int n, int mats) {
  return dc_align((size_t)n * (8 * kDcDoubles + 4 * kDcInts + kDcBytes)) + mats * dc_align((size_t)8 * n * n) + 256;
}
// Carves the arrays of a problem of order n; with Q == nullptr-sized matrices left out (leaf).
__host__ __device__ inline DcWork dc_vectors(char* base, int n) {
  DcWork W{};
  W.n = n;
  double* f = (double*)base;
  double** fs[] = {&W.D[0], &W.D[1], &W.ds, &W.zs, &W.dl, &W.w, &W.mu, &W.zh, &W.lam, &W.rc, &W.rs, &W.es};
  for (int i = 0; i < kDcDoubles; ++i) *fs[i] = f + (size_t)i * n;
  int* q = (int*)(f + (size_t)kDcDoubles * n);
  int** is[] = {&W.perm, &W.idx, &W.defl, &W.pos, &W.gat, &W.org, &W.rp, &W.rq, &W.dest};
  for (int i = 0; i < 9; ++i) *is[i] = q + (size_t)i * n;
  W.cnt = q + (size_t)9 * n;  // 4 n
  unsigned char* c = (unsigned char*)(q + (size_t)kDcInts * n);
  W.small = c;
  W.close = c + n;
  W.type = c + 2 * (size_t)n;
  return W;
}
// Q1, U: n x n doubles each elsewhere, or both null.
inline DcWork dc_carve(char* base, int n, double* Q1, double* U) {
  DcWork W = dc_vectors(base, n);
  char* p = base + dc_align((size_t)n * (8 * kDcDoubles + 4 * kDcInts + kDcBytes));
  auto take = [&](double* given) {
    if (given) return given;
    double* q = (double*)p;
    p += dc_align((size_t)8 * n * n);
    return q;
  };
  W.Q[0] = take(nullptr);
  W.Q[1] = take(Q1);
  W.U = take(U);
  W.bad = (int*)p;
  W.ex = W.bad + 1;
  return W;
}
// The arrays of problem b (every array a uniform stride of `stride` bytes further on).
__device__ inline DcWork dc_at(DcWork W, size_t off) {
  auto mv = [&](auto*& p) { p = (std::remove_reference_t<decltype(p)>)((char*)p + off); };
  mv(W.D[0]); mv(W.D[1]); mv(W.ds); mv(W.zs); mv(W.dl); mv(W.w); mv(W.mu); mv(W.zh); mv(W.lam); mv(W.rc); mv(W.rs);
  mv(W.perm); mv(W.idx); mv(W.defl); mv(W.pos); mv(W.gat); mv(W.org); mv(W.rp); mv(W.rq); mv(W.dest); mv(W.cnt);
  mv(W.small); mv(W.close); mv(W.type); mv(W.Q[0]); mv(W.Q[1]); mv(W.U); mv(W.bad); mv(W.es); mv(W.ex);
  return W;
}

// The merge of rows [s, mid) and [mid, t) of T with off-diagonal e (at mid - 1); input in D[cur].
__device__ inline dc::Merge dc_merge(const DcWork& W, int cur, int s, int mid, int t, double e) {
  dc::Merge M;
  M.m = t - s;
  M.n1 = mid - s;
  M.rho = 2.0 * fabs(e);
  M.sign = e < 0.0 ? -1.0 : 1.0;
  M.D = W.D[cur] + s;
  M.ds = W.ds + s; M.zs = W.zs + s; M.dl = W.dl + s; M.w = W.w + s; M.mu = W.mu + s; M.zh = W.zh + s;
  M.lam = W.lam + s; M.rc = W.rc + s; M.rs = W.rs + s;
  M.perm = W.perm + s; M.idx = W.idx + s; M.defl = W.defl + s; M.pos = W.pos + s; M.gat = W.gat + s;
  M.org = W.org + s; M.rp = W.rp + s; M.rq = W.rq + s; M.dest = W.dest + s;
  M.cnt = W.cnt + 4 * s;
  M.small = W.small + s; M.close = W.close + s; M.type = W.type + s;
  return M;
}

// Rotations of the deflated pairs applied to row i of Q's block (column q at Qb + q ldq).
__device__ inline void dc_rotate_row(const dc::Merge& M, double* Qb, int ldq, int i) {
  const int nr = M.cnt[3];
  for (int r = 0; r < nr; ++r) {
    double* x = Qb + (size_t)i + (size_t)M.rp[r] * ldq;
    double* y = Qb + (size_t)i + (size_t)M.rq[r] * ldq;
    const double a = *x, b = *y;
    *x = M.rc[r] * a + M.rs[r] * b;
    *y = M.rc[r] * b - M.rs[r] * a;
  }
}

// One merge by one group (a warp or a CTA of nw warps) on local arrays: Q's block is replaced.
// width: lanes per root, so that the roots of a merge fill the group's warps (an iteration's
// scalar FP64 work, ~40 instructions of 64 clocks, is then shared by 32 / width roots).
template <class G>
__device__ inline void dc_merge_local(const G& g, int w, int nw, int width, const dc::Merge& M, double* D, double* Dn,
                                      double* Qb, double* Qn, double* U, int ldq) {
  const Lanes L(width);
  const int m = M.m;
  dc::setup(g, M, Qb + M.n1 - 1, Qb + M.n1 + (size_t)M.n1 * ldq, ldq);
  const int K = M.cnt[0];
  for_items(L, w, nw, K, [&](int k, bool wr) {
    dc::root(L, K, k, wr, M.dl, M.w, M.rho, M.mu + k, M.org + k, M.lam + k);
  });
  for (int i = g.tid; i < m; i += g.size) dc_rotate_row(M, Qb, ldq, i);
  g.sync();
  for_items(L, w, nw, K, [&](int k, bool wr) { dc::zhat(L, K, k, wr, M.dl, M.w, M.mu, M.org, M.zh); });
  g.sync();
  for_items(L, w, nw, K, [&](int k, bool wr) { dc::ucol(L, K, k, wr, M.dl, M.zh, M.mu, M.org, M.pos, U, ldq); });
  for_items(L, w, nw, m, [&](int t, bool wr) { dc::place(L, M, K, t, wr); });
  g.sync();
  for (int u = g.tid; u < m * m; u += g.size) {
    const int i = u % m, j = u / m;
    double a = 0.0;
    if (j < K) {
      const int p0 = i < M.n1 ? 0 : M.cnt[1], p1 = i < M.n1 ? M.cnt[2] : K;
      for (int p = p0; p < p1; ++p) a = fma(Qb[(size_t)i + (size_t)M.gat[p] * ldq], U[(size_t)p + (size_t)j * ldq], a);
    } else {
      a = Qb[(size_t)i + (size_t)M.perm[M.defl[j - K]] * ldq];
    }
    Qn[(size_t)i + (size_t)M.dest[j] * ldq] = a;
    if (i == 0) Dn[M.dest[j]] = j < K ? M.lam[j] : M.ds[M.defl[j - K]];
  }
  g.sync();
  for (int u = g.tid; u < m * m; u += g.size) Qb[(size_t)(u % m) + (size_t)(u / m) * ldq] = Qn[(size_t)(u % m) + (size_t)(u / m) * ldq];
  for (int i = g.tid; i < m; i += g.size) D[i] = Dn[i];
  g.sync();
}

__host__ __device__ inline int dc_bound(int n, long long i, int depth) { return (int)((i * n) >> depth); }

// Eigensystem of the pair [x0 + |e|, e; e, x1 + |e|] (x: diagonal entries with e torn off), by one
// rotation: D ascending, vectors in q (ld ldq).
__device__ inline void dc_pair(double e, double* D, double* q, int ldq) {
  const double a = D[0] + fabs(e), b = D[1] + fabs(e);
  double c = 1.0, s = 0.0, t = 0.0;
  if (e != 0.0) {
    const double tau = (b - a) / (2.0 * e);
    t = copysign(1.0 / (fabs(tau) + sqrt(1.0 + tau * tau)), tau);
    c = 1.0 / sqrt(1.0 + t * t);
    s = t * c;
  }
  const double la = a - t * e, lb = b + t * e;  // of (c, -s) and (s, c)
  const bool swap = la > lb;
  D[0] = swap ? lb : la;
  D[1] = swap ? la : lb;
  q[0] = swap ? s : c;
  q[1] = swap ? c : -s;
  q[ldq] = swap ? c : s;
  q[ldq + 1] = swap ? -s : c;
}

// Leaf blockIdx.x of 2^depth (at most 32 rows): its eigensystem by merges from pairs of rows up,
// the merges of a level at once with 8, 4, 2 or 1 of the warps each.  Latency-bound: a chain of
// divisions and square roots per root.  l = 30: 252 -> 195 us against merges from single rows
// with one warp or the whole CTA each.
__global__ void __launch_bounds__(256) dc_leaf_kernel(int n, int depth, const double* d0,
                                                      const double* e0, int ld_de, DcWork W0,
                                                      size_t stride) {
  dep_wait(false);
  __shared__ double sQ[LEAF * LEAF], sQn[LEAF * LEAF], sU[LEAF * LEAF];
  __shared__ double s_red[8], s_e[LEAF];
  __shared__ long long s_max[8];
  __shared__ __align__(16) char s_vec[LEAF * (8 * kDcDoubles + 4 * kDcInts + kDcBytes)];
  const DcWork W = dc_at(W0, stride * blockIdx.y);
  const double* d = d0 + (size_t)blockIdx.y * ld_de;
  const double* e = e0 + (size_t)blockIdx.y * ld_de;
  const int s = dc_bound(n, blockIdx.x, depth), t = dc_bound(n, blockIdx.x + 1, depth), m = t - s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const DcWork V = dc_vectors(s_vec, LEAF);
  for (int u = tid; u < LEAF * LEAF; u += 256) sQ[u] = (u % LEAF == u / LEAF) ? 1.0 : 0.0;
  // 2^ex T: its largest entry, by every leaf for itself
  auto bits = [](double x) { return __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll; };
  long long mx = 0;
  for (int i = tid; i < n; i += 256) mx = max(mx, max(bits(d[i]), i + 1 < n ? bits(e[i]) : 0));
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_max[warp] = mx;
  __syncthreads();
  for (int w = 0; w < 8; ++w) mx = max(mx, s_max[w]);
  const int ex = dc::scale_of(__longlong_as_double(mx));
  if (blockIdx.x == 0 && tid == 0) *W.ex = ex;
  for (int i = tid; i < m; i += 256) {
    const int r = s + i;
    // every off-diagonal is torn at some level
    const double lo = r > 0 ? fabs(ldexp(e[r - 1], ex)) : 0.0, er = r + 1 < n ? ldexp(e[r], ex) : 0.0;
    V.D[0][i] = ldexp(d[r], ex) - lo - fabs(er);
    s_e[i] = er;
    W.es[r] = er;
    if (!isfinite(d[r]) || !isfinite(er)) *W.bad = 1;
  }
  __syncthreads();
  if (tid < 16) {  // single rows: at most one each side
    const long long i0 = ((long long)blockIdx.x << 5) + 2 * tid;
    const int a = dc_bound(n, i0, depth + 5) - s, b = dc_bound(n, i0 + 1, depth + 5) - s,
              c = dc_bound(n, i0 + 2, depth + 5) - s;
    if (b > a && c > b) dc_pair(s_e[b - 1], V.D[0] + a, sQ + a + a * LEAF, LEAF);
  }
  __syncthreads();
  for (int h = 3; h >= 0; --h) {
    const int nw = 8 >> h, q = warp / nw, wq = warp - q * nw;  // warps per merge, this warp's merge
    const long long i0 = ((long long)blockIdx.x << (h + 1)) + 2 * q;
    const int a = dc_bound(n, i0, depth + h + 1) - s, b = dc_bound(n, i0 + 1, depth + h + 1) - s,
              c = dc_bound(n, i0 + 2, depth + h + 1) - s;
    if (b > a && c > b) {  // (an empty half: nothing to merge)
      const dc::Merge M = dc_merge(V, 0, a, b, c, s_e[b - 1]);
      const int at = a + a * LEAF;
      if (h == 3)
        dc_merge_local(WarpGroup{lane, 32}, 0, 1, 8, M, V.D[0] + a, V.D[1] + a, sQ + at, sQn + at, sU + at, LEAF);
      else
        dc_merge_local(PartGroup{tid - 32 * nw * q, 32 * nw, 1 + q, s_red + nw * q}, wq, nw, 8, M, V.D[0] + a,
                       V.D[1] + a, sQ + at, sQn + at, sU + at, LEAF);
    }
    __syncthreads();
  }
  for (int u = tid; u < m * m; u += 256)
    W.Q[0][(size_t)(s + u % m) + (size_t)(s + u / m) * n] = sQ[(u % m) + (u / m) * LEAF];
  for (int i = tid; i < m; i += 256) W.D[0][s + i] = V.D[0][i];
}

// Merge blockIdx.(y or z) of the level with 2^depth blocks below it; cur: input buffer.
__device__ inline dc::Merge dc_level_merge(const DcWork& W, int cur, int depth, int q, int* s) {
  const int a = dc_bound(W.n, 2 * q, depth), b = dc_bound(W.n, 2 * q + 1, depth), c = dc_bound(W.n, 2 * q + 2, depth);
  *s = a;
  return dc_merge(W, cur, a, b, c, W.es[b - 1]);
}

__global__ void __launch_bounds__(512) dc_setup_kernel(DcWork W0, size_t stride, int cur, int depth) {
  dep_wait(false);
  __shared__ double red[16];
  const DcWork W = dc_at(W0, stride * blockIdx.y);
  int s;
  const dc::Merge M = dc_level_merge(W, cur, depth, blockIdx.x, &s);
  const double* Qb = W.Q[cur] + s + (size_t)s * W.n;
  dc::setup(CtaGroup{(int)threadIdx.x, 512, red}, M, Qb + M.n1 - 1, Qb + M.n1 + (size_t)M.n1 * W.n, W.n);
}

// phase 0: roots, and the rotations of Q's rows; 1: corrected z; 2: U and the new order.
__global__ void __launch_bounds__(128) dc_phase_kernel(DcWork W0, size_t stride, int cur, int depth, int phase) {
  dep_wait(false);
  const DcWork W = dc_at(W0, stride * blockIdx.z);
  int s;
  const dc::Merge M = dc_level_merge(W, cur, depth, blockIdx.y, &s);
  const Lanes L(32);
  const int w = blockIdx.x * 4 + (threadIdx.x >> 5), nw = gridDim.x * 4;
  const int K = M.cnt[0];
  if (phase == 0) {
    for (int k = w; k < K; k += nw) dc::root(L, K, k, true, M.dl, M.w, M.rho, M.mu + k, M.org + k, M.lam + k);
    double* Qb = W.Q[cur] + s + (size_t)s * W.n;
    for (int i = blockIdx.x * 128 + threadIdx.x; i < M.m; i += gridDim.x * 128) dc_rotate_row(M, Qb, W.n, i);
  } else if (phase == 1) {
    for (int k = w; k < K; k += nw) dc::zhat(L, K, k, true, M.dl, M.w, M.mu, M.org, M.zh);
  } else {
    double* Ub = W.U + s + (size_t)s * W.n;
    for (int k = w; k < K; k += nw) dc::ucol(L, K, k, true, M.dl, M.zh, M.mu, M.org, M.pos, Ub, W.n);
    for (int t = w; t < M.m; t += nw) dc::place(L, M, K, t, true);
  }
}

// Q_new[:, dest] = Q[:, gathered] U (64 x 32 tiles, FP64), deflated columns copied.
__global__ void __launch_bounds__(256) dc_gemm_kernel(DcWork W0, size_t stride, int cur, int depth, int parts) {
  dep_wait(false);
  const DcWork W = dc_at(W0, stride * (blockIdx.z / parts));
  int s;
  const dc::Merge M = dc_level_merge(W, cur, depth, blockIdx.z % parts, &s);
  constexpr int BK = 16;
  __shared__ double As[BK][64], Bs[BK][33];
  const int m0 = blockIdx.y * 64, j0 = blockIdx.x * 32, m = M.m, n1 = M.n1, K = M.cnt[0], ld = W.n;
  if (m0 >= m || j0 >= m) return;
  const double* Q = W.Q[cur] + s + (size_t)s * ld;
  const double* U = W.U + s + (size_t)s * ld;
  double* Qn = W.Q[cur ^ 1] + s + (size_t)s * ld;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double acc[4][2] = {};
  if (j0 < K) {
    const int p0 = m0 >= n1 ? M.cnt[1] : 0, p1 = m0 + 64 <= n1 ? M.cnt[2] : K;
    for (int pb = p0; pb < p1; pb += BK) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int i = tid & 63, k = (tid >> 6) + 4 * r;
        As[k][i] = (m0 + i < m && pb + k < p1) ? Q[(size_t)(m0 + i) + (size_t)M.gat[pb + k] * ld] : 0.0;
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int k = tid & 15, j = (tid >> 4) + 16 * r;
        Bs[k][j] = (j0 + j < K && pb + k < p1) ? U[(size_t)(pb + k) + (size_t)(j0 + j) * ld] : 0.0;
      }
      __syncthreads();
#pragma unroll
      for (int k = 0; k < BK; ++k) {
        double a[4], b[2];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = As[k][ty + 16 * i];
        b[0] = Bs[k][tx];
        b[1] = Bs[k][tx + 16];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          acc[i][0] = fma(a[i], b[0], acc[i][0]);
          acc[i][1] = fma(a[i], b[1], acc[i][1]);
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int j = j0 + tx + 16 * c;
    if (j >= m) continue;
    const int dj = M.dest[j];
    const double* src = j < K ? nullptr : Q + (size_t)M.perm[M.defl[j - K]] * ld;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = m0 + ty + 16 * i;
      if (r < m) Qn[(size_t)r + (size_t)dj * ld] = src ? src[r] : acc[i][c];
    }
    if (m0 == 0 && ty == 0) W.D[cur ^ 1][s + dj] = j < K ? M.lam[j] : M.ds[M.defl[j - K]];
  }
}

int dc_depth(int n) {
  int depth = 0;
  while (ceil_div(n, 1 << depth) > LEAF) ++depth;
  return depth;
}

// Eigensystems of `batch` tridiagonals (d, e at strides of ld_de) in the arrays W (strides of
// `stride` bytes); returns the buffer that holds D and Q in *cur.
int stedc(cudaStream_t st, int n, int batch, const double* d, const double* e, int ld_de, const DcWork& W,
          size_t stride, int* cur, int* launches) {
  for (int b = 0; b < batch; ++b) {
    // the flag lies behind Q[0], or behind Q[1] and U too
    const size_t span = (char*)W.bad - (char*)W.Q[0];
    CHASE_CUDA_TRY(cudaMemsetAsync((char*)W.Q[0] + stride * b, 0, span + sizeof(int), st));
    if (span < 2 * dc_align((size_t)8 * n * n))
      CHASE_CUDA_TRY(cudaMemsetAsync(W.Q[1], 0, (size_t)8 * n * n, st));
  }
  const int depth = dc_depth(n);
  launch_dep(st, dim3(1 << depth, batch), 256, 0, dc_leaf_kernel, n, depth, d, e, ld_de, W, stride);
  int nl = 1, c = 0;
  for (int h = depth; h > 0; --h) {
    const int parts = 1 << (h - 1), m = ceil_div(n, parts);  // rows of a merge, at most
    launch_dep(st, dim3(parts, batch), 512, 0, dc_setup_kernel, W, stride, c, h);
    for (int phase = 0; phase < 3; ++phase)
      launch_dep(st, dim3(ceil_div(m, 4), parts, batch), 128, 0, dc_phase_kernel, W, stride, c, h, phase);
    launch_dep(st, dim3(ceil_div(m, 32), ceil_div(m, 64), parts * batch), 256, 0, dc_gemm_kernel, W, stride, c, h,
               parts);
    nl += 5;
    c ^= 1;
  }
  *cur = c;
  if (launches) *launches += nl;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

// ---------------------------------------------------------------------------
// 3. Back-transformation
// ---------------------------------------------------------------------------
// 3. Back-transformation.  H_a ... H_{a+7} = I - V T V^H with an upper triangular T (8 x 8): block
// blockIdx.x of eight reflectors, T row by row into Tb.
constexpr int BTK = 8;
constexpr int BT_MIN = 24;  // rows from which the blocked form is used (l = 30 real: the same 25 us;
                            // l = 60 real 58 -> 26 us, l = 600 complex 3.5 -> 2.05 ms)

template <class T>
__global__ void __launch_bounds__(256) bt_factor_kernel(int l, const T* H, int ldh,
                                                        const T* tau, T* Tb) {
  dep_wait(false);
  __shared__ T G[BTK][BTK], S[BTK][BTK];
  const int a = blockIdx.x * BTK, kb = min(BTK, l - 1 - a), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x < BTK * BTK) S[threadIdx.x / BTK][threadIdx.x % BTK] = Sc<T>::zero();
  for (int u = warp; u < BTK * BTK; u += 8) {  // G[i][j] = v_i^H v_j, i < j
    const int i = u / BTK, j = u % BTK;
    if (i >= j || j >= kb) continue;
    T s = Sc<T>::zero();
    for (int r = a + j + 1 + lane; r < l; r += 32)
      Sc<T>::fmac(s, H[(size_t)r + (size_t)(a + i) * ldh], H[(size_t)r + (size_t)(a + j) * ldh]);
    s = warp_addt(s);
    if (lane == 0) G[i][j] = s;
  }
  __syncthreads();
  if (warp == 0) {
    for (int j = 0; j < kb; ++j) {  // column j: tau_j, above it -tau_j T G[:, j]
      const T t = tau[a + j];
      if (lane < j) {
        T s = Sc<T>::zero();
        for (int k = lane; k < j; ++k) Sc<T>::fma(s, S[lane][k], G[k][j]);
        S[lane][j] = Sc<T>::scale(Sc<T>::mul(t, s), -1.0);
      } else if (lane == j) {
        S[j][j] = t;
      }
      __syncwarp();
    }
    for (int u = lane; u < BTK * BTK; u += 32) Tb[(size_t)blockIdx.x * BTK * BTK + u] = S[u / BTK][u % BTK];
  }
}

__device__ __forceinline__ double sum8t(const double* s, int lane) { return sum8(s, lane); }
__device__ __forceinline__ z64 sum8t(const z64* s, int lane) {
  double re[8], im[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) { re[j] = s[j].x; im[j] = s[j].y; }
  return z64{sum8(re, lane), sum8(im, lane)};
}
__device__ __forceinline__ double shfl_t(double v, int src) { return __shfl_sync(0xffffffffu, v, src); }
__device__ __forceinline__ z64 shfl_t(z64 v, int src) { return z64{shfl_t(v.x, src), shfl_t(v.y, src)}; }

// Column c of W = H_0 H_1 ... H_{l-2} Z[:, c], eight reflectors at a time: z -= V (T (V^H z)).  One
// warp per column, z in shared memory, the next 32 rows of V loaded ahead of their use; dw = D (NaN
// if T was not finite).  FP64-bound (8 l^2 / 2 FMAs of a complex column on one sub-partition): one
// reflector at a time waited for each one's loads and for 10 additions of the warp's sum.
template <class T>
__global__ void __launch_bounds__(128) bt_block_kernel(int l, const T* H, int ldh,
                                                       const T* Tb, const double* Z,
                                                       const double* D, const int* bad, const int* ex, const int* ex0,
                                                       T* Wm, int ldw, double* dw) {
  dep_wait(false);
  extern __shared__ __align__(16) unsigned char bt_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x * (blockDim.x >> 5) + warp;
  if (c >= l) return;
  const bool nan_out = *bad != 0;
  T* z = (T*)bt_smem + (size_t)warp * l;
  for (int i = lane; i < l; i += 32) z[i] = Sc<T>::from_re(nan_out ? nan("") : Z[(size_t)i + (size_t)c * l]);
  if (lane == 0) dw[c] = nan_out ? nan("") : ldexp(D[c], -(*ex + *ex0));
  __syncwarp();
  const int nb = nan_out ? 0 : (l - 1 + BTK - 1) / BTK;
  for (int b = nb - 1; b >= 0; --b) {
    const int a = b * BTK, kb = min(BTK, l - 1 - a), r0 = (a + 1) & ~31;
    T x[BTK], y[BTK], s[BTK];
    auto load = [&](int i) {
#pragma unroll
      for (int j = 0; j < BTK; ++j)
        y[j] = (j < kb && i > a + j && i < l) ? H[(size_t)i + (size_t)(a + j) * ldh] : Sc<T>::zero();
    };
    const int ti = lane >> 2, tk = lane & 3;
    const T t0 = Tb[(size_t)b * BTK * BTK + ti * BTK + tk], t1 = Tb[(size_t)b * BTK * BTK + ti * BTK + tk + 4];
#pragma unroll
    for (int j = 0; j < BTK; ++j) s[j] = Sc<T>::zero();
    load(r0 + lane);
    for (int i = r0 + lane; i - lane < l; i += 32) {
#pragma unroll
      for (int j = 0; j < BTK; ++j) x[j] = y[j];
      if (i - lane + 32 < l) load(i + 32);
      const T zi = i < l ? z[i] : Sc<T>::zero();
#pragma unroll
      for (int j = 0; j < BTK; ++j) Sc<T>::fmac(s[j], x[j], zi);
    }
    load(r0 + lane);
    const T q = sum8t(s, lane);  // of reflector lane / 4
    T u = Sc<T>::mul(t0, shfl_t(q, 4 * tk));
    Sc<T>::fma(u, t1, shfl_t(q, 4 * (tk + 4)));
    u = Sc<T>::add(u, shfl_t(u, lane ^ 1));
    u = Sc<T>::scale(Sc<T>::add(u, shfl_t(u, lane ^ 2)), -1.0);
#pragma unroll
    for (int j = 0; j < BTK; ++j) s[j] = shfl_t(u, 4 * j);
    for (int i = r0 + lane; i - lane < l; i += 32) {
#pragma unroll
      for (int j = 0; j < BTK; ++j) x[j] = y[j];
      if (i - lane + 32 < l) load(i + 32);
      T zi = i < l ? z[i] : Sc<T>::zero();
#pragma unroll
      for (int j = 0; j < BTK; ++j) Sc<T>::fma(zi, x[j], s[j]);
      if (i < l) z[i] = zi;
    }
  }
  T* out = Wm + (size_t)c * ldw;
  for (int i = lane; i < l; i += 32) out[i] = z[i];
}

// The same one reflector at a time, for few rows and for columns that do not fit shared memory.
// Column c of W = H_0 H_1 ... H_{l-2} Z[:, c]: one warp per column, the column in shared memory
// (in_smem) or in place; dw = D (NaN if T was not finite).
template <class T>
__global__ void backtransform_kernel(int l, const T* H, int ldh, const T* tau,
                                     const double* Z, const double* D, const int* bad, const int* ex,
                                     const int* ex0, T* Wm, int ldw, double* dw, int in_smem) {
  dep_wait(false);
  extern __shared__ __align__(16) unsigned char bt_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.x * (blockDim.x >> 5) + warp;
  if (c >= l) return;
  T* out = Wm + (size_t)c * ldw;
  T* z = in_smem ? (T*)bt_smem + (size_t)warp * l : out;
  if (*bad) {
    for (int i = lane; i < l; i += 32) out[i] = Sc<T>::from_re(nan(""));
    if (lane == 0) dw[c] = nan("");
    return;
  }
  for (int i = lane; i < l; i += 32) z[i] = Sc<T>::from_re(Z[(size_t)i + (size_t)c * l]);
  if (lane == 0) dw[c] = ldexp(D[c], -(*ex + *ex0));
  __syncwarp();
  for (int j = l - 2; j >= 0; --j) {
    const T t = tau[j];
    if (Sc<T>::re(t) == 0.0 && im_of(t) == 0.0) continue;
    const T* v = H + (size_t)j * ldh;
    T s = Sc<T>::zero();
    for (int i = j + 1 + lane; i < l; i += 32) Sc<T>::fmac(s, v[i], z[i]);
    s = Sc<T>::scale(Sc<T>::mul(t, warp_addt(s)), -1.0);
    for (int i = j + 1 + lane; i < l; i += 32) {
      T x = z[i];
      Sc<T>::fma(x, v[i], s);
      z[i] = x;
    }
    __syncwarp();
  }
  if (in_smem)
    for (int i = lane; i < l; i += 32) out[i] = z[i];
}

// theta and squared first components of problem blockIdx.x (NaN if its T was not finite)
__global__ void dc_extract_kernel(DcWork W0, size_t stride, int cur, double* theta, double* weight) {
  dep_wait();
  const DcWork W = dc_at(W0, stride * blockIdx.x);
  for (int i = threadIdx.x; i < W.n; i += blockDim.x) {
    const double q = W.Q[cur][(size_t)i * W.n];
    theta[(size_t)blockIdx.x * W.n + i] = *W.bad ? nan("") : ldexp(W.D[cur][i], -*W.ex);
    weight[(size_t)blockIdx.x * W.n + i] = *W.bad ? nan("") : q * q;
  }
}
// problems of one pass over the tridiagonals: as many as fit about 128 MB, at least one
int tridiag_pass(int m, int batch) {
  return (int)std::max<size_t>(1, std::min<size_t>(batch, ((size_t)128 << 20) / dc_align(dc_bytes(m, 3))));
}

struct EighLayout {
  size_t tau, d, e, xb, cb, part, scr, tb, ex, dc, total;
};
// Shared memory of the reduction: partial sums and factors of the own columns, three vectors.
size_t tri_fixed_smem(int l, int own, size_t elem) { return elem * (6 * (size_t)own + 3 * (size_t)l); }
bool tri_vec_smem(int l, size_t elem) { return tri_fixed_smem(l, ceil_div(l, kNumSMs), elem) <= kSmemMax - 1024; }
EighLayout eigh_layout(int l, size_t elem) {
  EighLayout L{};
  size_t off = 0;
  auto take = [&](size_t b) { const size_t o = off; off += dc_align(b); return o; };
  L.tau = take(elem * l);
  L.d = take(8 * (size_t)l);
  L.e = take(8 * (size_t)l);
  L.xb = take(2 * elem * l);
  L.cb = take(2 * elem * l);
  L.part = take(2 * 8 * kNumSMs);
  L.scr = take(tri_vec_smem(l, elem) ? 0 : elem * 3 * (size_t)l * kNumSMs);
  L.tb = take(sizeof(GridBar));
  L.ex = take(sizeof(int));
  L.dc = take(dc_bytes(l, 1));
  L.total = off;
  return L;
}

template <class T>
int tridiag(cudaStream_t st, int l, T* H, int ldh, char* base, const EighLayout& L, DevStatus* dst,
            int* launches) {
  T *tau = (T*)(base + L.tau), *xb = (T*)(base + L.xb), *cb = (T*)(base + L.cb);
  double *d = (double*)(base + L.d), *e = (double*)(base + L.e), *part = (double*)(base + L.part);
  GridBar* gb = (GridBar*)(base + L.tb);
  int* ex = (int*)(base + L.ex);
  // CTAs: one for every 1000 elements (complex: x 4), one alone below 3000, where a column's
  // FP64 work costs less than the grid barrier (measured: l = 30 real 0.142 ms on one CTA, 0.171
  // on four; l = 60 real 0.417 and 0.343; l = 230 complex 1.95 on 38, 1.73 on 76)
  const double work = (double)l * l * (Sc<T>::cplx ? 4.0 : 1.0);
  int G = work < 3000.0 ? 1 : (int)std::min<double>(kNumSMs, work / 1000.0);
  const bool vec = tri_vec_smem(l, sizeof(T));
  if (!vec) G = kNumSMs;
  G = std::max(1, std::min(G, l));
  size_t smem;
  for (;; ++G) {  // (fewer CTAs own more columns each)
    smem = vec ? tri_fixed_smem(l, ceil_div(l, G), sizeof(T)) : sizeof(T) * 6 * (size_t)ceil_div(l, G);
    if (smem <= kSmemMax - 1024 || G >= std::min(l, kNumSMs)) break;
  }
  if (smem > kSmemMax - 1024) return CHASE_ERR_UNSUPPORTED;
  T* scr = vec ? nullptr : (T*)(base + L.scr);
  const size_t cols = sizeof(T) * (size_t)ceil_div(l, G) * l;
  int in_smem = smem + cols <= kSmemMax - 1024;
  if (in_smem) smem += cols;
  CHASE_CUDA_TRY(cudaFuncSetAttribute((const void*)tridiag_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kSmemMax - 1024));
  CHASE_CUDA_TRY(cudaMemsetAsync(gb, 0, sizeof(GridBar), st));
  void* args[] = {(void*)&l,  (void*)&H,  (void*)&ldh,  (void*)&in_smem, (void*)&tau, (void*)&d,  (void*)&e,
                  (void*)&xb, (void*)&cb, (void*)&part, (void*)&scr,     (void*)&ex,  (void*)&gb,
                  (void*)&dst};
  CHASE_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)tridiag_kernel<T>, dim3(G), dim3(TNT), args, smem, st));
  if (launches) ++*launches;
  return 0;
}

}  // namespace

size_t eigh_work_bytes(int l, size_t elem) { return eigh_layout(l, elem).total; }

template <class T>
int eigh(cudaStream_t st, int l, T* H, int ldh, T* W, int ldw, double* dw, T* spare, void* work, size_t work_bytes,
         DevStatus* dst, int* launches) {
  if (l <= 0) return 0;
  const EighLayout L = eigh_layout(l, sizeof(T));
  if (L.total > work_bytes) return CHASE_ERR_OOM;
  if (ldw != l) return CHASE_ERR_UNSUPPORTED;
  char* base = (char*)work;
  T* tau = (T*)(base + L.tau);
  double *d = (double*)(base + L.d), *e = (double*)(base + L.e);
  const int* ex0 = (const int*)(base + L.ex);
  TRY_EIG(tridiag<T>(st, l, H, ldh, base, L, dst, launches));
  // (the eigenvectors' place holds U until they are formed)
  const DcWork D = dc_carve(base + L.dc, l, (double*)spare, (double*)W);
  int cur = 0;
  TRY_EIG(stedc(st, l, 1, d, e, 0, D, 0, &cur, launches));
  const int wpc = (int)std::max<size_t>(1, std::min<size_t>(4, (kSmemMax - 1024) / (sizeof(T) * (size_t)l)));
  const size_t smem = sizeof(T) * (size_t)l * wpc;
  const int in_smem = smem <= kSmemMax - 1024;
  CHASE_CUDA_TRY(cudaFuncSetAttribute((const void*)backtransform_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)kSmemMax - 1024));
  if (in_smem && l >= BT_MIN) {
    T* Tb = (T*)D.Q[cur ^ 1];  // free by now: l^2 doubles for 8 (l + 7) elements
    launch_dep(st, ceil_div(l - 1, BTK), 256, 0, bt_factor_kernel<T>, l, H, ldh, tau, Tb);
    CHASE_CUDA_TRY(cudaFuncSetAttribute((const void*)bt_block_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)kSmemMax - 1024));
    launch_dep(st, ceil_div(l, wpc), 32 * wpc, smem, bt_block_kernel<T>, l, H, ldh, Tb, D.Q[cur], D.D[cur], D.bad,
               D.ex, ex0, W, ldw, dw);
    if (launches) ++*launches;
  } else {
    launch_dep(st, ceil_div(l, wpc), 32 * wpc, in_smem ? smem : 0, backtransform_kernel<T>, l, H, ldh, tau, D.Q[cur],
               D.D[cur], D.bad, D.ex, ex0, W, ldw, dw, in_smem);
  }
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

size_t tridiag_work_bytes(int m, int batch) { return dc_align(dc_bytes(m, 3)) * tridiag_pass(m, batch); }

int tridiag_eigs(cudaStream_t st, int m, int batch, const double* alpha, const double* beta, double* theta,
                 double* weight, void* work, size_t work_bytes, int* launches) {
  if (m <= 0 || batch <= 0) return 0;
  if (tridiag_work_bytes(m, batch) > work_bytes) return CHASE_ERR_OOM;
  const size_t stride = dc_align(dc_bytes(m, 3));
  const DcWork W = dc_carve((char*)work, m, nullptr, nullptr);
  for (int r = 0, nb = tridiag_pass(m, batch); r < batch; r += nb) {
    const int cnt = std::min(nb, batch - r);
    int cur = 0;
    TRY_EIG(stedc(st, m, cnt, alpha + (size_t)r * m, beta + (size_t)r * m, m, W, stride, &cur, launches));
    launch_dep(st, cnt, 128, 0, dc_extract_kernel, W, stride, cur, theta + (size_t)r * m, weight + (size_t)r * m);
    if (launches) ++*launches;
  }
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

template int eigh<double>(cudaStream_t, int, double*, int, double*, int, double*, double*, void*, size_t, DevStatus*, int*);
template int eigh<z64>(cudaStream_t, int, z64*, int, z64*, int, double*, z64*, void*, size_t, DevStatus*, int*);

}  // namespace chase
