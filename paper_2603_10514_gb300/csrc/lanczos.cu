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
// Column c of A and every q_r become integers relative to their largest entry (x 2^{55 - e},
// |x| < 2^e, rounded), cut into two halves of 28 bits with sign; their products are summed exactly
// in 64 bits, three per pair (the middle one from the sums of halves).  GB300 has 2 FP64 FMAs per
// clock per SM, but 16 multiply-adds of 32 x 32 + 64 bits, so three of these cost less than half
// of one.  The entries are rounded to 2^-56 of the column's and the vector's largest, the sums
// only at the end, where the FP64 sums they replace round every term.
constexpr int kLzBits = 55, kLzBad = 1 << 20;  // exponent of a column with NaN or infinity

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
template <bool EVEN>
__device__ __forceinline__ void lz_split(double x, int e, int* hi, int* lo) {
  const long long b = __double_as_longlong(x);
  const int ex = (int)(b >> 52) & 0x7FF;
  // x = m 2^{ex - 1075}, so x 2^{55 - e} = 4 m 2^{-d}; v: 8 m
  const unsigned long long v = (((unsigned long long)b & ((1ull << 52) - 1)) | (ex ? 1ull << 52 : 0ull)) << 3;
  const int d = min(max(1077 - kLzBits + e - max(ex, 1), 0), 63);
  const unsigned long long u = v >> d;
  unsigned long long r = (u + 1) >> 1;
  if (EVEN && (u & 1) && (u << d) == v) r &= ~1ull;
  int h = (int)(r >> 28), l = (int)((uint32_t)r & 0xFFFFFFFu);
  const int up = l >> 27, s = (int)(b >> 63);
  h += up;
  l -= up << 28;
  *hi = (h ^ s) - s;
  *lo = (l ^ s) - s;
}
template <bool EVEN>
__device__ __forceinline__ int2 lz_cut(double x, int e) {
  int2 v;
  lz_split<EVEN>(x, e, &v.x, &v.y);
  return v;
}
template <bool EVEN>
__device__ __forceinline__ int4 lz_cut(z64 x, int e) {
  int4 v;
  lz_split<EVEN>(x.x, e, &v.x, &v.y);
  lz_split<EVEN>(x.y, e, &v.z, &v.w);
  return v;
}
template <class T> struct LzInt { using type = int2; };
template <> struct LzInt<z64> { using type = int4; };

// Exponents of the columns of A (n x n), one warp each, and the largest of them.
template <class T>
__global__ void __launch_bounds__(256) lz_colexp_kernel(int n, const T* A, int lda,
                                                        int* ea, int* emax) {
  dep_wait();
  const int lane = threadIdx.x & 31, c = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (c >= n) return;
  const T* col = A + (size_t)c * lda;
  long long m = 0;
#pragma unroll 8
  for (int i = lane; i < n; i += 32) m = max(m, lz_abs(col[i]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) {
    const int e = lz_exp(m);
    ea[c] = e;
    if (m > 0 && e < kLzBad) atomicMax(emax, e);
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
// A's column c with q_r -- one warp for KC columns, A read once for all runs in full lines; Qi, eq:
// the q_r cut up.  A term of x is at most 2^56 (complex: two): the sums of a lane are taken out
// after 120 (60) terms.  Bound by the wide multiply-adds.  Real n = 8000, 4 runs: FP64 465 us a
// step -> 252 us.
template <class T, int R, int KC>
__global__ void __launch_bounds__(256) lz_product_kernel(int n, const T* A, int lda,
                                                         const int* ea,
                                                         const typename LzInt<T>::type* Qi,
                                                         const int* eq, const int* emax, T* W) {
  dep_wait();
  constexpr int NP = Sc<T>::cplx ? 2 : 1, NV = KC * R * NP;
  const int lane = threadIdx.x & 31, c0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * KC;
  if (c0 >= n) return;
  const T* col[KC];
  int e[KC];
#pragma unroll
  for (int k = 0; k < KC; ++k) {
    const int c = min(c0 + k, n - 1);
    col[k] = A + (size_t)c * lda;
    e[k] = ea[c];
  }
  const int em = lz_scale(*emax);
  double sum[NV];
#pragma unroll
  for (int u = 0; u < NV; ++u) sum[u] = 0.0;
  constexpr int CHUNK = 32 * (Sc<T>::cplx ? 60 : 120);
  for (int i0 = 0; i0 < n; i0 += CHUNK) {
    LzSum s[NV];
#pragma unroll
    for (int u = 0; u < NV; ++u) s[u] = LzSum{0, 0, 0};
    const int i1 = min(n, i0 + CHUNK);
#pragma unroll 4
    for (int i = i0 + lane; i < i1; i += 32) {
      typename LzInt<T>::type q[R];
#pragma unroll
      for (int r = 0; r < R; ++r) q[r] = Qi[(size_t)r * n + i];
#pragma unroll
      for (int k = 0; k < KC; ++k) {
        const auto a = lz_cut<false>(col[k][i], e[k]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          LzSum* p = s + (k * R + r) * NP;
          p->add(a.x, a.y, q[r].x, q[r].y);
          if constexpr (Sc<T>::cplx) {  // conj(a) q
            p[0].add(a.z, a.w, q[r].z, q[r].w);
            p[1].add(a.x, a.y, q[r].z, q[r].w);
            p[1].add(-a.z, -a.w, q[r].x, q[r].y);
          }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < NV; ++u) sum[u] += s[u].value();
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
      const int k = u / (R * NP), r = u / NP % R, x = e[k] + eq[r];
      if (c0 + k < n)
        ((double*)W)[((size_t)r * n + c0 + k) * NP + u % NP] =
            x >= kLzBad / 2 ? nan("") : scalbn(sum[u], x - em - 2 * kLzBits);
    }
}

template <class T, int R>
void lz_launch(cudaStream_t st, int n, const T* A, int lda, const int* ea, const typename LzInt<T>::type* Qi,
               const int* eq, const int* emax, T* W) {
  constexpr int KC = Sc<T>::cplx ? 1 : 2;
  launch_dep(st, ceil_div(n, 8 * KC), 256, 0, lz_product_kernel<T, R, KC>, n, A, lda, ea, Qi, eq, emax, W);
}

template <class T>
int lz_product(cudaStream_t st, int n, int nruns, const T* A, int lda, const int* ea,
               const typename LzInt<T>::type* Qi, const int* eq, const int* emax, T* W,
               int* nl) {
  for (int r = 0; r < nruns; r += 4) {
    const auto* q = Qi + (size_t)r * n;
    T* w = W + (size_t)r * n;
    switch (std::min(4, nruns - r)) {
      case 1: lz_launch<T, 1>(st, n, A, lda, ea, q, eq + r, emax, w); break;
      case 2: lz_launch<T, 2>(st, n, A, lda, ea, q, eq + r, emax, w); break;
      case 3: lz_launch<T, 3>(st, n, A, lda, ea, q, eq + r, emax, w); break;
      default: lz_launch<T, 4>(st, n, A, lda, ea, q, eq + r, emax, w); break;
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
                                                            int m, int j, typename LzInt<T>::type* qi, int* eq,
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
    qi[(size_t)r * n + i] = lz_cut<true>(q, e);
  }
}

}  // namespace

template <class T>
int lanczos_bounds(cudaStream_t st, int n, const T* A, int lda, int nruns, const T* V0, int ldv,
                   int m, int ell, double* out, void* work, size_t work_bytes, int* launches) {
  // workspace: basis (m + 1) x n x nruns | W n x nruns | coef nruns x (m + 1) | alpha, beta |
  //            theta, weights | q_j cut up | exponents | work of the tridiagonal eigensolver
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
  int* ea = (int*)(base + off); off += al(sizeof(int) * ((size_t)n + nruns + 1));
  int *eq = ea + n, *emax = eq + nruns;
  if (off > work_bytes) return CHASE_ERR_OOM;
  int nl = 0;
  CHASE_CUDA_TRY(cudaMemsetAsync(emax, 0x80, sizeof(int), st));
  // q_0 = v / ||v|| for every run
  TRY_LZ(copy_cols<T>(st, n, nruns, V0, ldv, W, n, &nl));
  launch_dep(st, ceil_div(n, 8), 256, 0, lz_colexp_kernel<T>, n, A, lda, ea, emax);
  launch_dep(st, nruns, 512, 0, lz_normalize_kernel<T>, n, W, Qb, beta, m, 0, Qi, eq,
             Qb, pstride, 0, alpha);  // beta[.,0] rewritten below
  nl += 2;
  const int blocks = (int)std::min<size_t>((pstride + 255) / 256, (size_t)kNumSMs * 16);
  for (int j = 0; j < m; ++j) {
    // W = A q_j (up to four runs per pass over A)
    TRY_LZ(lz_product<T>(st, n, nruns, A, lda, ea, Qi, eq, emax, W, &nl));
    // coefficients against q_0..q_j: coef[., j] is alpha_j; subtracting all of them is the
    // three-term step plus full re-orthogonalisation (classical Gram-Schmidt, twice)
    for (int pass = 0; pass < 2; ++pass) {
      launch_dep(st, dim3(nruns, j + 1), 256, 0, lz_dots_kernel<T>, n, Qb, pstride, W, coef, m + 1);
      if (pass == 0) launch_dep(st, 1, 32, 0, lz_store_alpha_kernel<T>, nruns, coef, m + 1, j, alpha, m);
      launch_dep(st, blocks, 256, 0, lz_sub_kernel<T>, n, nruns, Qb, pstride, W, coef, m + 1, j + 1);
      nl += (pass == 0) ? 3 : 2;
    }
    launch_dep(st, nruns, 512, 0, lz_normalize_kernel<T>, n, W, Qb + (size_t)(j + 1) * pstride, beta, m, j, Qi, eq,
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
         4 * al(8 * (size_t)nruns * m) + al(elem * ps) + al(4 * ((size_t)n + nruns + 1)) + tridiag_work_bytes(m, nruns);
}

template int lanczos_bounds<double>(cudaStream_t, int, const double*, int, int, const double*, int,
                                    int, int, double*, void*, size_t, int*);
template int lanczos_bounds<z64>(cudaStream_t, int, const z64*, int, int, const z64*, int, int, int,
                                 double*, void*, size_t, int*);

}  // namespace chase
