// gemm_fp64.cu -- FP64 (real and complex) dense products with a fused
// three-term epilogue, for the Chebyshev filter (Algorithm 4), the Gram
// matrices of CholeskyQR (Algorithm 2), the triangular step X R^{-1} and the
// Rayleigh-Ritz products (Algorithm 1).
//
//   C[i,j] = alpha * sum_k op(A)[i,k] B[k,j] + beta * X[i,j] + gamma * Y[i,j]
//
// op(A) = A or A^H.  X and Y may alias C: each element of X / Y is read by the
// thread that then writes the same element of C, which is what lets the filter
// write V_i over V_{i-2} in place.
//
// GB300 issues 2 FP64 FMAs per SM per clock (~1.2 TFLOP/s for the whole GPU, measured), so a warp's
// FP64 instruction holds its sub-partition for 64 clocks and nothing else binds these products:
// not HBM, not shared memory.  What counts is that every sub-partition has the same number of
// them and that none is spent on padding.
//   - Tiles of 64 rows by up to 64 columns, the columns shared out evenly over the tiles.  A warp
//     takes 32 rows and every fourth column, so a tile costs its own columns, not a multiple of
//     16 or 32; the odd columns fall on other sub-partitions in every second CTA.
//   - One wave of two CTAs per SM, each with the same number of single K steps, over tile borders
//     (gemm_split.h): no last wave.  Tiles shared by CTAs have their parts summed in a fixed order
//     by a second kernel, which applies the epilogue.
// Against tiles of 64 x 32 (64 x 16) cut into equal K chunks, a step of the filter: n = 1531 complex,
// 57 columns 1022 -> 903 us (the pipe alone: 916 at 1.92 GHz), 33 columns 1016 -> 535, 17 columns
// 536 -> 293; n = 1000 real, 1 column 63 -> 23, 30 columns 106 -> 80; n = 5000 complex, 300 columns
// 54.8 -> 48.8 ms.
#include "common.cuh"
#include "gemm_split.h"
#include "kernels.h"

#include <utility>

namespace chase {

namespace {

constexpr int BM = kGemmRows;
constexpr int BK = 8;
constexpr int NT = 256;
constexpr int TN = kGemmCols / 4;  // columns of a thread (one row)

// acc[j] += sum over kn steps of K of a b[4 j], j < nc: a loop of its own for every nc, since an
// FP64 instruction that is predicated off holds the pipe as long as one that is not.
template <class T, int NC>
__device__ __forceinline__ void block_fma_n(const T* a, const T* b, int kn, T* acc) {
#pragma unroll 2
  for (int kk = 0; kk < kn; ++kk) {
    const T x = a[kk * (BM + 1)];
#pragma unroll
    for (int j = 0; j < NC; ++j) Sc<T>::fma(acc[j], x, b[kk * kGemmCols + 4 * j]);
  }
}
template <class T, int... J>
__device__ __forceinline__ void block_fma(std::integer_sequence<int, J...>, int nc, const T* a, const T* b, int kn,
                                          T* acc) {
  (void)((nc == J + 1 && (block_fma_n<T, J + 1>(a, b, kn, acc), true)) || ...);
}

template <class T, bool TRANS_A>
__global__ void __launch_bounds__(NT, 2) gemm_kernel(GemmSplit sp, const T* __restrict__ A, int lda,
                                                     const T* __restrict__ B, int ldb, T* C, int ldc,
                                                     double alpha, double beta, const T* X, int ldx,
                                                     double gamma, const T* Y, int ldy,
                                                     T* __restrict__ partial) {
  __shared__ T As[2][BK][BM + 1];
  __shared__ T Bs[2][BK][kGemmCols];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = blockIdx.x;
  const int row = 32 * (warp & 1) + lane;
  const int grp = ((warp >> 1) + g + g / kNumSMs) & 3;  // first column: rotated, see above
  long long w = sp.whole ? 0 : sp.begin(g);
  const long long w1 = sp.whole ? 0 : sp.begin(g + 1);
  do {
    const GemmTile t = sp.whole ? sp.tile(g) : sp.at(w);
    const int kb = sp.whole ? 0 : (int)(w - t.w0);
    const int ke = sp.whole ? t.kt : (int)min((long long)t.kt, kb + (w1 - w));
    const int nc = (t.nb - grp + 3) >> 2;
    T acc[TN];
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[j] = Sc<T>::zero();

    T ra[2], rb[2];  // the next block of K
    auto load = [&](int k0) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int i = TRANS_A ? (tid >> 3) + 32 * r : tid & 63;
        const int ka = k0 + (TRANS_A ? tid & 7 : (tid >> 6) + 4 * r), gi = t.m0 + i;
        ra[r] = Sc<T>::zero();
        if (gi < sp.M && ka < ke)
          ra[r] = TRANS_A ? Sc<T>::conj(A[(size_t)ka + (size_t)gi * lda]) : A[(size_t)gi + (size_t)ka * lda];
        const int j = (tid >> 3) + 32 * r, kk = k0 + (tid & 7);
        rb[r] = Sc<T>::zero();
        if (j < t.nb && kk < ke) rb[r] = B[(size_t)kk + (size_t)(t.n0 + j) * ldb];
      }
    };
    int s = 0;
    if (kb < ke) load(kb);
    for (int k0 = kb; k0 < ke; k0 += BK, s ^= 1) {
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        if (TRANS_A) As[s][tid & 7][(tid >> 3) + 32 * r] = ra[r];
        else As[s][(tid >> 6) + 4 * r][tid & 63] = ra[r];
        Bs[s][tid & 7][(tid >> 3) + 32 * r] = rb[r];
      }
      __syncthreads();  // (the other buffer is written only after this block's barrier: one is enough)
      if (k0 + BK < ke) load(k0 + BK);
      block_fma<T>(std::make_integer_sequence<int, TN>(), nc, &As[s][0][row], &Bs[s][0][grp], min(BK, ke - k0), acc);
    }
    __syncthreads();  // before the next tile's first block

    if (ke - kb < t.kt) {
      T* P = partial + (long long)(g + t.t) * sp.slot_elems();
#pragma unroll
      for (int j = 0; j < TN; ++j)
        if (j < nc) P[(grp + 4 * j) * BM + row] = acc[j];
    } else {
      const int gi = t.m0 + row;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int gj = t.n0 + grp + 4 * j;
        if (j < nc && gi < sp.M && !(sp.upper && gi > gj)) {
          T v = Sc<T>::scale(acc[j], alpha);
          if (beta != 0.0) v = Sc<T>::add(v, Sc<T>::scale(X[(size_t)gi + (size_t)gj * ldx], beta));
          if (gamma != 0.0) v = Sc<T>::add(v, Sc<T>::scale(Y[(size_t)gi + (size_t)gj * ldy], gamma));
          C[(size_t)gi + (size_t)gj * ldc] = v;
        }
      }
    }
    w += ke - kb;
  } while (w < w1);
}

// Sums the parts of the tiles that CTAs shared, in their order, and applies the epilogue.
// blockIdx.x: tile, blockIdx.y: columns y, y + gridDim.y, ...
template <class T>
__global__ void __launch_bounds__(128) split_reduce_kernel(GemmSplit sp, const T* __restrict__ partial, T* C,
                                                           int ldc, double alpha, double beta, const T* X, int ldx,
                                                           double gamma, const T* Y, int ldy) {
  const GemmTile t = sp.tile(blockIdx.x);
  const int g0 = sp.owner(t.w0), g1 = sp.owner(t.w0 + t.kt - 1);
  if (g0 == g1) return;
  const int row = threadIdx.x & 63, gi = t.m0 + row;
  if (gi >= sp.M) return;
  for (int j = 2 * blockIdx.y + (threadIdx.x >> 6); j < t.nb; j += 2 * gridDim.y) {
    const int gj = t.n0 + j;
    if (sp.upper && gi > gj) continue;
    const T* p = partial + j * BM + row;
    T v = p[(g0 + t.t) * sp.slot_elems()];
    for (int g = g0 + 1; g <= g1; ++g) v = Sc<T>::add(v, p[(g + t.t) * sp.slot_elems()]);
    v = Sc<T>::scale(v, alpha);
    if (beta != 0.0) v = Sc<T>::add(v, Sc<T>::scale(X[(size_t)gi + (size_t)gj * ldx], beta));
    if (gamma != 0.0) v = Sc<T>::add(v, Sc<T>::scale(Y[(size_t)gi + (size_t)gj * ldy], gamma));
    C[(size_t)gi + (size_t)gj * ldc] = v;
  }
}

}  // namespace

template <class T>
int gemm(cudaStream_t st, bool transA, int M, int N, int K, const T* A, int lda, const T* B,
         int ldb, T* C, int ldc, double alpha, double beta, const T* X, int ldx, double gamma,
         const T* Y, int ldy, Scratch scratch, bool upper_only, bool tri_b, int* launches) {
  if (M <= 0 || N <= 0) return 0;
  // kmin: a CTA with fewer K steps of a tile costs about as much to start as it computes (a step is
  // up to 2 us in complex arithmetic, 0.5 in real; a launch and the second kernel ~3)
  const GemmSplit sp = gemm_split(M, N, K, upper_only, tri_b, 2 * kNumSMs, Sc<T>::cplx ? 8 : 16,
                                  (long long)(scratch.bytes / sizeof(T)));
  T* partial = sp.whole ? nullptr : (T*)scratch.ptr;
  if (transA)
    gemm_kernel<T, true><<<sp.G, NT, 0, st>>>(sp, A, lda, B, ldb, C, ldc, alpha, beta, X, ldx, gamma, Y, ldy,
                                              partial);
  else
    gemm_kernel<T, false><<<sp.G, NT, 0, st>>>(sp, A, lda, B, ldb, C, ldc, alpha, beta, X, ldx, gamma, Y, ldy,
                                               partial);
  if (launches) ++*launches;
  if (!sp.whole) {
    split_reduce_kernel<T><<<dim3(sp.T, std::max(1, ceil_div(sp.bn, 8))), 128, 0, st>>>(
        sp, partial, C, ldc, alpha, beta, X, ldx, gamma, Y, ldy);
    if (launches) ++*launches;
  }
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

template int gemm<double>(cudaStream_t, bool, int, int, int, const double*, int, const double*,
                          int, double*, int, double, double, const double*, int, double,
                          const double*, int, Scratch, bool, bool, int*);
template int gemm<z64>(cudaStream_t, bool, int, int, int, const z64*, int, const z64*, int, z64*,
                       int, double, double, const z64*, int, double, const z64*, int, Scratch, bool,
                       bool, int*);

}  // namespace chase
