// lanczos.cu -- spectral bounds for the filter by a few Lanczos runs
// (Algorithm 1: "estimate lambda_1, lambda_ell and lambda_n").
//
// nruns runs advance together: one product A * [q_1 ... q_nruns] per step,
// column-wise alpha / beta, full re-orthogonalisation of each run's new vector
// against its own basis, then the m x m tridiagonals of all runs are
// diagonalised together (eigh.cu).  The host only reduces the m * nruns Ritz
// values and weights to the three bounds:
//   b_sup      = max_r (theta_max^r + |beta_m^r|)   -- an upper bound of lambda_n
//   lambda1    = min_r theta_min^r
//   lambda_ell = smallest pooled Ritz value where the spectral-density estimate
//                (n / nruns) sum_r sum_{theta_i^r <= x} tau_i^r reaches ell
// (tau_i^r: squared first component of the i-th eigenvector of run r's T).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <numeric>
#include <type_traits>
#include <vector>

#include "../../include/chase_gb300.h"
#include "common.cuh"
#include "kernels.h"

#define TRY_LZ(x)            \
  do {                       \
    int _rc = (x);           \
    if (_rc) return _rc;     \
  } while (0)

namespace chase {

namespace {

__device__ inline float warp_sumf(float v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ inline double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <class T>
__device__ inline T block_sum_t(T v, double* red);

template <>
__device__ inline double block_sum_t<double>(double v, double* red) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double t = 0.0;
  for (int i = 0; i < nw; ++i) t += red[i];
  return t;
}

template <>
__device__ inline z64 block_sum_t<z64>(z64 v, double* red) {
  const double a = block_sum_t<double>(v.x, red);
  const double b = block_sum_t<double>(v.y, red);
  return z64{a, b};
}

// ---- products A q in fixed point ----
// Column c of A (its diagonal entry apart) and every q_r become integers relative to their largest
// entry (x 2^{55 - e}, |x| < 2^e, rounded), cut into two halves of 28 bits with sign; their products
// are summed exactly in 64 bits, three per pair (the middle one from the sums of halves).  GB300 has
// 2 FP64 FMAs per clock per SM, but 16 multiply-adds of 32 x 32 + 64 bits, so three of these cost
// less than half of one.  Entries far below the largest of their column or vector lose bits that FP64
// keeps, but the sums are rounded only at the end, where FP64 rounds every term.  With a, b the
// entries over the largest ones' powers of two, the sum's error is, in the mean square,
//   2^-56 / sqrt 3 sqrt(sum a^2 + sum b^2)            in fixed point, and about
//   2^-53 sqrt(5.3 + 1700 / n) / 20.4 sum |a b|       in FP64 (chains of n / 32 terms, 5 more sums,
//                                                       terms of either sign: less than for one sign);
// every column of every step is checked for the first being the smaller.  Where it is not (sparse
// columns, columns and vectors with large and small entries at different places) the column is summed
// in FP64, for the rest of the call.
constexpr int kLzBits = 55, kLzBad = 1 << 20;  // exponent of a column with NaN or infinity
constexpr int kLzFp64 = -kLzBad;               // of one that is summed in FP64

__device__ __forceinline__ long long lz_abs(double x) { return __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll; }
__device__ __forceinline__ long long lz_abs(z64 a) { return max(lz_abs(a.x), lz_abs(a.y)); }

// smallest e >= -1021 with |x| < 2^e for the bits of the largest |x| (subnormal numbers stay exact)
__device__ __forceinline__ int lz_exp(long long bits) {
  if (bits >= 0x7FF0000000000000ll) return kLzBad;
  if (bits == 0) return 0;
  int e;
  frexp(__longlong_as_double(bits), &e);
  return max(e, -1021);
}

// x 2^{55 - e} rounded: hi 2^28 + lo with |hi| <= 2^27, |lo| <= 2^27.  EVEN: ties to even, for the
// vectors; the matrix saves the instructions (ties away from zero, in the last of 56 bits).
// top: |x| 2^{23 - e}, truncated.
template <bool EVEN>
__device__ __forceinline__ void lz_split(double x, int e, int* hi, int* lo, uint32_t* top) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7FF;
  // x = m 2^{ex - 1075}, so x 2^{55 - e} = 4 m 2^{-d}; v: 8 m
  const unsigned long long v = (((unsigned long long)b & ((1ull << 52) - 1)) | (ex ? 1ull << 52 : 0ull)) << 3;
  const int d = min(max(1077 - kLzBits + e - max(ex, 1), 0), 63);
  const unsigned long long u = v >> d;
  unsigned long long r = (u + 1) >> 1;
  if (EVEN && (u & 1) && (u << d) == v) r &= ~1ull;
  *top = (uint32_t)(r >> 32);
  int h = (int)(r >> 28), l = (int)((uint32_t)r & 0xFFFFFFFu);
  const int up = l >> 27, s = (int)(b >> 63);
  h += up;
  l -= up << 28;
  *hi = (h ^ s) - s;
  *lo = (l ^ s) - s;
}
template <bool EVEN>
__device__ __forceinline__ int2 lz_cut(double x, int e, uint32_t* top) {
  int2 v;
  lz_split<EVEN>(x, e, &v.x, &v.y, top);
  return v;
}
template <bool EVEN>
__device__ __forceinline__ int4 lz_cut(z64 x, int e, uint32_t* top) {
  int4 v;
  lz_split<EVEN>(x.x, e, &v.x, &v.y, top);
  lz_split<EVEN>(x.y, e, &v.z, &v.w, top + 1);
  return v;
}
template <class T> struct LzInt { using type = int2; };
template <> struct LzInt<z64> { using type = int4; };
// The magnitudes for the check as floats, from integers up to 2^23.  Those of q: four runs of a row
// (complex: of its real, then its imaginary parts) in 16 bytes.
__device__ __forceinline__ float lz_mag(uint32_t top) { return __uint_as_float(0x4B000000u | top) - 8388608.0f; }
template <class T>
__host__ __device__ inline size_t lz_mags(int n) { return (size_t)n * (Sc<T>::cplx ? 8 : 4); }  // of four runs
__device__ __forceinline__ float2 lz_fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
      "fma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}

// Exponents of the columns of A (n x n), one warp each, without the diagonal entry (which is far
// above the others in many matrices), and the largest of them with it.
template <class T>
__global__ void __launch_bounds__(256) lz_colexp_kernel(int n, const T* A, int lda,
                                                        int* ea, int* emax) {
  dep_wait();
  const int lane = threadIdx.x & 31, c = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (c >= n) return;
  const T* col = A + (size_t)c * lda;
  long long m = 0;
#pragma unroll 8
  for (int i = lane; i < n; i += 32) m = max(m, i == c ? 0 : lz_abs(col[i]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    ea[c] = lz_exp(m);
    m = max(m, lz_abs(col[c]));
    if (m > 0 && lz_exp(m) < kLzBad) atomicMax(emax, lz_exp(m));
  }
}
// The runs advance with 2^-em A, whose entries are below 1: at the ends of FP64's range its residuals
// and their products would be subnormal or overflow.  emax starts far below any exponent.
__host__ __device__ inline int lz_scale(int emax) { return emax < -kLzBad ? 0 : emax; }

// Sums of products of high halves, low halves, and sums of halves.
struct LzSum {
  long long h, l, x;
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
    h += (long long)ah * bh;
    l += (long long)al * bl;
    x += (long long)(ah + al) * (bh + bl);
  }
  __device__ __forceinline__ double value() const {
    return fma(fma((double)h, 268435456.0, (double)(x - h - l)), 268435456.0, (double)l);
  }
};

// W[:, r] = 2^-em A q_r for R runs: A is Hermitian, so entry c of the product is the dot product of
// A's column c with q_r -- one warp per column, A read once for all runs in full lines; Q, Qi, Qm, eq:
// the q_r, cut up, their magnitudes, their exponents.  A term of x is at most 2^56 (complex: two): the
// sums of a lane are taken out after 120 (60) terms.  Bound by the wide multiply-adds, the instructions
// that cut A up and the loads of q from L2.  4 runs, 25 steps of n = 8000: real 12.8 ms in FP64 -> 7.7
// (7.2 without the check, two columns to a warp), complex 21.5; a sparse real matrix, in FP64, 13.4.
// Two blocks per SM, since more columns at once spread the reads of A over more pages (three: 11 ms).
template <class T, int R>
__global__ void __launch_bounds__(256, 2) lz_product_kernel(int n, const T* A, int lda,
                                                            int* ea, const T* Q,
                                                            const typename LzInt<T>::type* Qi,
                                                            const float4* Qm, const int* eq,
                                                            const int* emax, T* W) {
  dep_wait();
  constexpr bool Z = Sc<T>::cplx;
  constexpr int NP = Z ? 2 : 1, NV = R * NP, NR = (R + 1) / 2;
  const int lane = threadIdx.x & 31, c = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (c >= n) return;
  const T* col = A + (size_t)c * lda;
  const int e = ea[c], em = lz_scale(*emax);
  double sum[NV];
#pragma unroll
  for (int u = 0; u < NV; ++u) sum[u] = 0.0;
  // the check's sums: of a^2, and of |a b| for two runs each (a, b: over 2^-23)
  float sa = 0.0f;
  float2 sab[NP][NR];
#pragma unroll
  for (int h = 0; h < NP; ++h)
#pragma unroll
    for (int t = 0; t < NR; ++t) sab[h][t] = make_float2(0.0f, 0.0f);
  LzSum s[NV];
  // row i's terms of every sum; plain: neither the diagonal's nor past the end
  auto terms = [&](int i, auto plain) {
    const bool in = decltype(plain)::value || i < n;
    const int j = in ? i : 0;
    typename LzInt<T>::type q[R];
#pragma unroll
    for (int r = 0; r < R; ++r) q[r] = Qi[(size_t)r * n + j];
    float2 b[NP][2];
#pragma unroll
    for (int h = 0; h < NP; ++h) {
      const float4 v = Qm[j * NP + h];
      b[h][0] = make_float2(v.x, v.y);
      b[h][1] = make_float2(v.z, v.w);
    }
    T x = col[j];
    if (!decltype(plain)::value && (!in || j == c)) x = Sc<T>::zero();
    uint32_t top[2];
    const auto a = lz_cut<false>(x, e, top);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      LzSum* p = s + r * NP;
      p->add(a.x, a.y, q[r].x, q[r].y);
      if constexpr (Z) {  // conj(a) q
        p[0].add(a.z, a.w, q[r].z, q[r].w);
        p[1].add(a.x, a.y, q[r].z, q[r].w);
        p[1].add(-a.z, -a.w, q[r].x, q[r].y);
      }
    }
    const float f = lz_mag(top[0]);
    const float2 ff = make_float2(f, f);
    sa = fmaf(f, f, sa);
#pragma unroll
    for (int t = 0; t < NR; ++t) sab[0][t] = lz_fma2(ff, b[0][t], sab[0][t]);
    if constexpr (Z) {
      const float g = lz_mag(top[1]);
      const float2 gg = make_float2(g, g);
      sa = fmaf(g, g, sa);
#pragma unroll
      for (int t = 0; t < NR; ++t) {
        sab[0][t] = lz_fma2(gg, b[1][t], sab[0][t]);
        sab[1][t] = lz_fma2(ff, b[1][t], lz_fma2(gg, b[0][t], sab[1][t]));
      }
    }
  };
  constexpr int CHUNK = 32 * (Z ? 60 : 120), UNROLL = Z ? 2 : 8, ROWS = 32 * UNROLL;
  bool exact = e != kLzFp64;
  for (int i0 = 0; i0 < n && exact; i0 += CHUNK) {
#pragma unroll
    for (int u = 0; u < NV; ++u) s[u] = LzSum{0, 0, 0};
    const int i1 = min(n, i0 + CHUNK);
    for (int i = i0; i < i1; i += ROWS) {
      if (i + ROWS <= i1 && (c < i || c >= i + ROWS)) {
#pragma unroll
        for (int d = 0; d < UNROLL; ++d) terms(i + 32 * d + lane, std::true_type());
      } else {
#pragma unroll 1
        for (int j = i; j < min(i1, i + ROWS); j += 32) terms(j + lane, std::false_type());
      }
    }
#pragma unroll
    for (int u = 0; u < NV; ++u) sum[u] += s[u].value();
  }
  // sum a^2 + sum b^2 <= (2.4 + 780 / terms) (sum |a b|)^2; |q| = 1, so sum b^2 = 4^-eq
  const float a2 = warp_sumf(sa) * 0x1p-46f, lim = 2.4f + 780.0f / (float)(NP * n);
  bool ok = true;
#pragma unroll
  for (int u = 0; u < NV; ++u) {
    const int r = u / NP;
    const float2 v = sab[u % NP][r / 2];
    const float ab = warp_sumf(r % 2 ? v.y : v.x) * 0x1p-46f, b2 = exp2f(-2.0f * (float)max(eq[r], -50));
    ok = ok && a2 + b2 <= lim * ab * ab;
  }
  exact = exact && (ok || a2 == 0.0f);  // (0: nothing beside the diagonal entry, or NaN)
  const double scale = scalbn(1.0, -em);
  if (!exact) {
    if (lane == 0) ea[c] = kLzFp64;
#pragma unroll
    for (int u = 0; u < NV; ++u) sum[u] = 0.0;
    // (the scale after the sums, unless they might leave FP64's range: 1 FP64 instruction in 5)
    const bool late = abs(em) < 400;
    auto fp64 = [&](auto scaled) {
#pragma unroll 4
      for (int i = lane; i < n; i += 32) {
        T a = i == c ? Sc<T>::zero() : col[i];
        if (decltype(scaled)::value) a = Sc<T>::scale(a, scale);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const T q = Q[(size_t)r * n + i];
          if constexpr (Z) {
            z64 v{sum[2 * r], sum[2 * r + 1]};
            Sc<T>::fmac(v, a, q);
            sum[2 * r] = v.x;
            sum[2 * r + 1] = v.y;
          } else {
            Sc<T>::fmac(sum[r], a, q);
          }
        }
      }
    };
    if (late) fp64(std::false_type());
    else fp64(std::true_type());
    if (late) {
#pragma unroll
      for (int u = 0; u < NV; ++u) sum[u] *= scale;
    }
  }
  if constexpr (NV == 8) {  // lane 4 u gets sum u
    const double v = sum8(sum, lane);
#pragma unroll
    for (int u = 0; u < 8; ++u) sum[u] = __shfl_sync(0xffffffffu, v, 4 * u);
  } else {
#pragma unroll
    for (int u = 0; u < NV; ++u) sum[u] = warp_sum(sum[u]);
  }
#pragma unroll
  for (int u = 0; u < NV; ++u)
    if (lane == u) {
      const int r = u / NP, x = e + eq[r];
      double w = !exact ? sum[u] : x >= kLzBad / 2 ? nan("") : scalbn(sum[u], x - em - 2 * kLzBits);
      const T a = Sc<T>::scale(col[c], scale), q = Q[(size_t)r * n + c];
      if constexpr (Z) w = u % 2 ? fma(a.x, q.y, fma(-a.y, q.x, w)) : fma(a.x, q.x, fma(a.y, q.y, w));
      else w = fma(a, q, w);
      ((double*)W)[((size_t)r * n + c) * NP + u % NP] = w;
    }
}

template <class T, int R>
void lz_launch(cudaStream_t st, int n, const T* A, int lda, int* ea, const T* Q, const typename LzInt<T>::type* Qi,
               const float4* Qm, const int* eq, const int* emax, T* W) {
  launch_dep(st, ceil_div(n, 8), 256, 0, lz_product_kernel<T, R>, n, A, lda, ea, Q, Qi, Qm, eq, emax, W);
}

template <class T>
int lz_product(cudaStream_t st, int n, int nruns, const T* A, int lda, int* ea,
               const T* Q, const typename LzInt<T>::type* Qi, const float4* Qm, const int* eq, const int* emax,
               T* W, int* nl) {
  for (int r = 0; r < nruns; r += 4) {
    const T* q = Q + (size_t)r * n;
    const auto* qi = Qi + (size_t)r * n;
    const float4* qm = Qm + r / 4 * (lz_mags<T>(n) / 4);
    T* w = W + (size_t)r * n;
    switch (std::min(4, nruns - r)) {
      case 1: lz_launch<T, 1>(st, n, A, lda, ea, q, qi, qm, eq + r, emax, w); break;
      case 2: lz_launch<T, 2>(st, n, A, lda, ea, q, qi, qm, eq + r, emax, w); break;
      case 3: lz_launch<T, 3>(st, n, A, lda, ea, q, qi, qm, eq + r, emax, w); break;
      default: lz_launch<T, 4>(st, n, A, lda, ea, q, qi, qm, eq + r, emax, w); break;
    }
    ++*nl;
  }
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

// coef[r * ldc + p] = q_p^r^H w_r for p = 0..np-1 (one CTA per (r, p)); the basis of run r's
// step p is Qb + p * pstride + r * n.
template <class T>
__global__ void __launch_bounds__(256) lz_dots_kernel(int n, const T* Qb,
                                                      size_t pstride, const T* W,
                                                      T* coef, int ldc) {
  dep_wait();
  __shared__ double red[8];
  const int r = blockIdx.x, p = blockIdx.y;
  const T* q = Qb + (size_t)p * pstride + (size_t)r * n;
  const T* w = W + (size_t)r * n;
  T s = Sc<T>::zero();
  for (int i = threadIdx.x; i < n; i += 256) Sc<T>::fmac(s, q[i], w[i]);
  s = block_sum_t<T>(s, red);
  if (threadIdx.x == 0) coef[(size_t)r * ldc + p] = s;
}

// w_r -= sum_{p < np} coef[r, p] q_p^r   (elementwise, one thread per (i, r))
template <class T>
__global__ void lz_sub_kernel(int n, int nruns, const T* Qb, size_t pstride, T* W,
                              const T* coef, int ldc, int np) {
  dep_wait();
  const size_t total = (size_t)n * nruns;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % n), r = (int)(t / n);
    T w = W[t];
    for (int p = 0; p < np; ++p)
      w = Sc<T>::sub(w, Sc<T>::mul(coef[(size_t)r * ldc + p], Qb[(size_t)p * pstride + (size_t)r * n + i]));
    W[t] = w;
  }
}

// alpha_r = Re(coef[r, j]) (the Rayleigh quotient of step j), stored for the tridiagonal.
template <class T>
__global__ void lz_store_alpha_kernel(int nruns, const T* coef, int ldc, int j, double* alpha,
                                      int m) {
  dep_wait();
  const int r = threadIdx.x;
  if (r < nruns) alpha[r * m + j] = Sc<T>::re(coef[(size_t)r * ldc + j]);
}

// A number in (-1, 1) from a counter.
__device__ __forceinline__ double lz_random(uint32_t x) {
  x ^= x >> 16; x *= 0x7FEB352Du;
  x ^= x >> 15; x *= 0x846CA68Bu;
  x ^= x >> 16;
  return ((double)x + 0.5) * 0x1p-31 - 1.0;
}

// beta_r = ||w_r||; q_{j+1}^r = w_r / beta_r (one CTA per run), and its integers and exponent.  Where
// nothing is left of w_r beside the terms that it was reduced by (np > 0 basis vectors at Qb), the
// basis spans an invariant subspace and w_r has no direction of its own, least of all one orthogonal
// to the basis: beta_r = 0 then, and the run goes on from a pseudo-random vector orthogonal to it.
template <class T>
__global__ void __launch_bounds__(512) lz_normalize_kernel(int n, T* W, T* qn, double* beta,
                                                            int m, int j, typename LzInt<T>::type* qi, float* qm,
                                                            int* eq,
                                                            const T* Qb, size_t pstride, int np, const double* alpha) {
  dep_wait();
  __shared__ double red[16];
  __shared__ long long redm[16];
  const int r = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T* w = W + (size_t)r * n;
  long long mx;
  int ew;
  double scale, b;  // b = ||w|| 2^-ew: 1 / ||w|| may be out of range
  auto measure = [&]() {
    mx = 0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) mx = max(mx, lz_abs(w[i]));
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    __syncthreads();
    if (lane == 0) redm[warp] = mx;
    __syncthreads();
    for (int i = 0; i < (int)blockDim.x >> 5; ++i) mx = max(mx, redm[i]);
    // squares of w 2^-ew neither overflow nor underflow
    ew = lz_exp(mx) == kLzBad ? 0 : lz_exp(mx);
    scale = scalbn(1.0, -ew);
    double s = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) s += Sc<T>::abs2(Sc<T>::scale(w[i], scale));
    b = sqrt(block_sum_t<double>(s, red));
  };
  measure();
  bool ended = false;
  if (np > 0) {
    const double left = fabs(alpha[r * m + j]) + (j > 0 ? fabs(beta[r * m + j - 1]) : 0.0);
    ended = scalbn(b, ew) <= 0x1p-50 * left;
  }
  if (ended) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const uint32_t k = ((uint32_t)i * 64 + (uint32_t)r * 2) ^ ((uint32_t)j << 24);
      if constexpr (Sc<T>::cplx) w[i] = z64{lz_random(k), lz_random(k + 1)};
      else w[i] = lz_random(k);
    }
    for (int p = 0; p < 2 * np; ++p) {
      const T* q = Qb + (size_t)(p % np) * pstride + (size_t)r * n;
      T c = Sc<T>::zero();
      for (int i = threadIdx.x; i < n; i += blockDim.x) Sc<T>::fmac(c, q[i], w[i]);
      c = block_sum_t<T>(c, red);
      for (int i = threadIdx.x; i < n; i += blockDim.x) w[i] = Sc<T>::sub(w[i], Sc<T>::mul(c, q[i]));
    }
    measure();
  }
  if (threadIdx.x == 0) beta[r * m + j] = ended ? 0.0 : scalbn(b, ew);
  const double inv = (b > 0.0) ? 1.0 / b : 0.0;
  // the largest |q| is the largest |w| 2^-ew times inv (rounding keeps order)
  const int e = lz_exp(lz_abs(__longlong_as_double(mx) * scale * inv));
  if (threadIdx.x == 0) eq[r] = e;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const T q = Sc<T>::scale(Sc<T>::scale(w[i], scale), inv);
    qn[(size_t)r * n + i] = q;
    uint32_t top[2];
    qi[(size_t)r * n + i] = lz_cut<true>(q, e, top);
    float* mag = qm + r / 4 * lz_mags<T>(n) + (size_t)i * (Sc<T>::cplx ? 8 : 4) + r % 4;
    mag[0] = lz_mag(top[0]);
    if (Sc<T>::cplx) mag[4] = lz_mag(top[1]);
  }
}

}  // namespace

template <class T>
int lanczos_bounds(cudaStream_t st, int n, const T* A, int lda, int nruns, const T* V0, int ldv,
                   int m, int ell, double* out, void* work, size_t work_bytes, int* launches) {
  // workspace: basis (m + 1) x n x nruns | W n x nruns | coef nruns x (m + 1) | alpha, beta |
  //            theta, weights | q_j cut up, its magnitudes | exponents | work of the tridiagonal eigensolver
  auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t pstride = (size_t)n * nruns;
  size_t off = 0;
  char* base = (char*)work;
  T* Qb = (T*)(base + off); off += al(sizeof(T) * pstride * (m + 1));
  T* W = (T*)(base + off); off += al(sizeof(T) * pstride);
  T* coef = (T*)(base + off); off += al(sizeof(T) * (size_t)nruns * (m + 1));
  double* alpha = (double*)(base + off); off += al(sizeof(double) * (size_t)nruns * m);
  double* beta = (double*)(base + off); off += al(sizeof(double) * (size_t)nruns * m);
  double* th = (double*)(base + off); off += al(sizeof(double) * (size_t)nruns * m);
  double* tw = (double*)(base + off); off += al(sizeof(double) * (size_t)nruns * m);
  using I = typename LzInt<T>::type;
  I* Qi = (I*)(base + off); off += al(sizeof(I) * pstride);
  float* Qm = (float*)(base + off); off += al(4 * lz_mags<T>(n) * ((nruns + 3) / 4));
  int* ea = (int*)(base + off); off += al(sizeof(int) * ((size_t)n + nruns + 1));
  int *eq = ea + n, *emax = eq + nruns;
  if (off > work_bytes) return CHASE_ERR_OOM;
  int nl = 0;
  CHASE_CUDA_TRY(cudaMemsetAsync(emax, 0x80, sizeof(int), st));
  // q_0 = v / ||v|| for every run
  TRY_LZ(copy_cols<T>(st, n, nruns, V0, ldv, W, n, &nl));
  launch_dep(st, ceil_div(n, 8), 256, 0, lz_colexp_kernel<T>, n, A, lda, ea, emax);
  launch_dep(st, nruns, 512, 0, lz_normalize_kernel<T>, n, W, Qb, beta, m, 0, Qi, Qm, eq,
             Qb, pstride, 0, alpha);  // beta[.,0] rewritten below
  nl += 2;
  const int blocks = (int)std::min<size_t>((pstride + 255) / 256, (size_t)kNumSMs * 16);
  for (int j = 0; j < m; ++j) {
    // W = A q_j (up to four runs per pass over A)
    TRY_LZ(lz_product<T>(st, n, nruns, A, lda, ea, Qb + (size_t)j * pstride, Qi, (const float4*)Qm, eq, emax, W,
                         &nl));
    // coefficients against q_0..q_j: coef[., j] is alpha_j; subtracting all of them is the
    // three-term step plus full re-orthogonalisation (classical Gram-Schmidt, twice)
    for (int pass = 0; pass < 2; ++pass) {
      launch_dep(st, dim3(nruns, j + 1), 256, 0, lz_dots_kernel<T>, n, Qb, pstride, W, coef, m + 1);
      if (pass == 0) launch_dep(st, 1, 32, 0, lz_store_alpha_kernel<T>, nruns, coef, m + 1, j, alpha, m);
      launch_dep(st, blocks, 256, 0, lz_sub_kernel<T>, n, nruns, Qb, pstride, W, coef, m + 1, j + 1);
      nl += (pass == 0) ? 3 : 2;
    }
    launch_dep(st, nruns, 512, 0, lz_normalize_kernel<T>, n, W, Qb + (size_t)(j + 1) * pstride, beta, m, j, Qi, Qm,
               eq,
               Qb, pstride, j + 1, alpha);
    ++nl;
  }
  // Ritz values and weights of each run
  std::vector<double> hth((size_t)nruns * m), htau((size_t)nruns * m), hbeta((size_t)nruns * m);
  TRY_LZ(tridiag_eigs(st, m, nruns, alpha, beta, th, tw, base + off, work_bytes - off, &nl));
  CHASE_CUDA_TRY(cudaMemcpyAsync(hth.data(), th, sizeof(double) * (size_t)nruns * m, cudaMemcpyDeviceToHost, st));
  CHASE_CUDA_TRY(cudaMemcpyAsync(htau.data(), tw, sizeof(double) * (size_t)nruns * m, cudaMemcpyDeviceToHost, st));
  CHASE_CUDA_TRY(cudaMemcpyAsync(hbeta.data(), beta, sizeof(double) * (size_t)nruns * m,
                                 cudaMemcpyDeviceToHost, st));
  int em = 0;
  CHASE_CUDA_TRY(cudaMemcpyAsync(&em, emax, sizeof(int), cudaMemcpyDeviceToHost, st));
  CHASE_CUDA_TRY(cudaStreamSynchronize(st));
  em = lz_scale(em);
  for (double& t : hth) t = std::ldexp(t, em);
  for (double& b : hbeta) b = std::ldexp(b, em);
  double bsup = -1e300, l1 = 1e300;
  for (int r = 0; r < nruns; ++r) {
    const double* t = hth.data() + (size_t)r * m;
    bsup = std::max(bsup, t[m - 1] + std::fabs(hbeta[(size_t)r * m + m - 1]));
    l1 = std::min(l1, t[0]);
  }
  std::vector<int> ord((size_t)nruns * m);
  std::iota(ord.begin(), ord.end(), 0);
  std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return hth[a] < hth[b]; });
  double cum = 0.0, lell = hth[ord.back()];
  for (int idx : ord) {
    cum += htau[idx] * (double)n / (double)nruns;
    if (cum >= (double)ell * (1.0 - 1e-10)) { lell = hth[idx]; break; }  // up to rounding
  }
  out[0] = l1;
  out[1] = std::max(lell, l1);
  out[2] = bsup;
  if (launches) *launches += nl;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

size_t lanczos_work_bytes(size_t elem, int n, int nruns, int m) {
  auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t ps = (size_t)n * nruns;
  return al(elem * ps * (m + 1)) + al(elem * ps) + al(elem * (size_t)nruns * (m + 1)) +
         4 * al(8 * (size_t)nruns * m) + al(elem * ps) +
         al(4 * (elem == sizeof(z64) ? lz_mags<z64>(n) : lz_mags<double>(n)) * ((nruns + 3) / 4)) + al(4 * ((size_t)n + nruns + 1)) + tridiag_work_bytes(m, nruns);
}

template int lanczos_bounds<double>(cudaStream_t, int, const double*, int, int, const double*, int,
                                    int, int, double*, void*, size_t, int*);
template int lanczos_bounds<z64>(cudaStream_t, int, const z64*, int, int, const z64*, int, int, int,
                                 double*, void*, size_t, int*);

}  // namespace chase
