// chol_trsm.cu -- the small ell x ell factorisation of CholeskyQR (Algorithm 2:
// R = chol(X^H X); Algorithm 3: chol(R + sI)) and the inverse of the triangular factor used
// for X <- X R^{-1}.
//
// Cholesky: one cooperative kernel over blocks of 32 rows.  Per block
//   A  CTA 0 factors the diagonal block, eliminating [G_kk | I] so that M = R_kk^{-H} comes
//      with it, and publishes both (a flag);
//   B  block row R_k. = M G_k., one warp per column;
//   C  trailing update G -= R_k.^H R_k. of the upper triangle, one warp per 8 x 8 tile;
// with a grid barrier after B and after C.  A non-positive or non-finite pivot j is reported as
// info = j + 1 in the device status word (LAPACK convention) and every CTA leaves.  The
// kernel reads G through L2 only (other CTAs wrote it).
//
// Inverse: CTA b takes columns b and n - 1 - b of R^{-1} (together every CTA the same work),
// each by back substitution over the same blocks of 32, with the M of step A for the diagonal
// blocks: no division and three block barriers per 32 rows.
//
// What binds is FP64 at 2 FMAs per clock per SM (a warp instruction takes 64 clocks of a
// sub-partition) and, in A, the chain of pivots: blocks of 32 keep A's share on one SM short
// (64 would take four times that: the FP64 work of a block grows with its cube), the rest is
// spread over all SMs.  n = 600 complex: 4.8 -> 2.0 ms (1.62 factor, 0.41 inverse) against blocks
// of 64 in separate launches and an inverse by single columns; n = 30 real 57 -> 26 us.
#include "../../include/chase_gb300.h"
#include "common.cuh"
#include "kernels.h"

namespace chase {

namespace {

constexpr int CB = 32;              // rows of a block
constexpr int CT = 8;               // trailing tiles are 8 x 8
constexpr int CNT = 256, CW = CNT / 32;
constexpr int CLD = CB + 1;
constexpr int kSmemMax = 227 * 1024;

struct CholBar {
  GridBar bar;
  unsigned ready;  // diagonal blocks factored
  int fail;        // a pivot was not positive
  int pad[2];
};

template <class T> __device__ __forceinline__ T ld_cg(const T* p);
template <> __device__ __forceinline__ double ld_cg<double>(const double* p) { return __ldcg(p); }
template <> __device__ __forceinline__ z64 ld_cg<z64>(const z64* p) {
  const double2 v = __ldcg((const double2*)p);
  return z64{v.x, v.y};
}

// A: factors the b x b block at `off` (CTA 0, CNT threads).  B, M: CB x CLD in shared memory.
// Returns false (on every thread) after a failing pivot, reported in dst.
template <class T>
__device__ bool chol_block(int b, T* G, int ldg, int off, double shift, T* B, T* M, T* Mb, DevStatus* dst) {
  __shared__ int s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) s_fail = 0;
  for (int t = tid; t < CB * CB; t += CNT) {
    const int i = t % CB, j = t / CB;
    T g = Sc<T>::zero();
    if (i <= j && j < b) g = ld_cg(G + (size_t)(off + i) + (size_t)(off + j) * ldg);
    if (i == j) g = Sc<T>::add(g, Sc<T>::from_re(shift));
    B[i * CLD + j] = g;
    M[i * CLD + j] = i == j ? Sc<T>::one() : Sc<T>::zero();
  }
  __syncthreads();
  // row p of [B | M] minus conj(R[j][p]) times row j
  auto eliminate = [&](int j, int p) {
    const T f = Sc<T>::scale(Sc<T>::conj(B[j * CLD + p]), -1.0);
    if (lane >= p) Sc<T>::fma(B[p * CLD + lane], f, B[j * CLD + lane]);
    else if (lane <= j) Sc<T>::fma(M[p * CLD + lane], f, M[j * CLD + lane]);
  };
  // pivot of row j, and the row scaled by it (one warp)
  auto pivot = [&](int j) {
    const double d = Sc<T>::re(B[j * CLD + j]);
    const bool bad = !(d > 0.0) || !isfinite(d);
    const double r = bad ? 1.0 : rsqrt(d);
    __syncwarp();
    if (lane > j) B[j * CLD + lane] = Sc<T>::scale(B[j * CLD + lane], r);
    else M[j * CLD + lane] = Sc<T>::scale(M[j * CLD + lane], r);
    if (lane == 0 && bad) {
      s_fail = 1;
      atomicCAS(&dst->chol_info, 0, off + j + 1);
    }
  };
  // Warp 0 runs ahead with the next row and its pivot, while the warps of the other
  // sub-partitions eliminate from the rows after it (warp 4 shares warp 0's FP64 pipe and idles).
  if (warp == 0) pivot(0);
  __syncthreads();
  if (s_fail) return false;
  for (int j = 0; j + 1 < b; ++j) {
    if (warp == 0) {
      eliminate(j, j + 1);
      __syncwarp();
      pivot(j + 1);
    } else if (warp != 4) {
      for (int p = j + 1 + (warp < 4 ? warp : warp - 1); p < b; p += 6) eliminate(j, p);
    }
    __syncthreads();
    if (s_fail) return false;
  }
  for (int t = tid; t < CB * CB; t += CNT) {
    const int i = t % CB, j = t / CB;
    // (the diagonal of B holds the pivots: their roots are taken here, off the chain)
    const T r = B[i * CLD + j];
    if (i <= j && j < b)
      G[(size_t)(off + i) + (size_t)(off + j) * ldg] = i == j ? Sc<T>::from_re(sqrt(Sc<T>::re(r))) : r;
    Mb[t] = (i < b && j <= i) ? M[i * CLD + j] : Sc<T>::zero();  // column-major CB x CB
  }
  return true;
}

// G (n x n, upper triangle) -> R in place; Mb: the blocks' R_kk^{-H}.  Rinv is written here when
// n <= CB (one block).
template <class T>
__global__ void __launch_bounds__(CNT) chol_kernel(int n, T* G, int ldg, double shift_factor, T* Mb, T* Rinv,
                                                   int ldri, CholBar* cb, DevStatus* dst) {
  extern __shared__ __align__(16) unsigned char chol_smem[];
  T* sm = (T*)chol_smem;
  __shared__ int s_ok;
  __shared__ double s_red[CW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G_ = gridDim.x, gw = blockIdx.x * CW + warp, nw = G_ * CW;
  unsigned bars = 0;
  double shift = 0.0;
  if (shift_factor > 0.0 && blockIdx.x == 0) {
    // s = shift_factor ||X||_F^2 with ||X||_F^2 = trace(X^H X), before anything is updated
    double tr = 0.0;
    for (int j = tid; j < n; j += CNT) tr += Sc<T>::re(ld_cg(G + (size_t)j + (size_t)j * ldg));
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if (lane == 0) s_red[warp] = tr;
    __syncthreads();
    for (int w = 0; w < CW; ++w) shift += s_red[w];
    shift *= shift_factor;
  }
  for (int kb = 0, off = 0; off < n; ++kb, off += CB) {
    const int b = min(CB, n - off), rest = n - off - b;
    T* Mk = Mb + (size_t)kb * CB * CB;
    if (blockIdx.x == 0) {
      const bool ok = chol_block<T>(b, G, ldg, off, shift, sm, sm + CB * CLD, Mk, dst);
      __syncthreads();
      if (tid == 0) {
        if (!ok) atomicExch(&cb->fail, 1);
        asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(&cb->ready), "r"(kb + 1) : "memory");
      }
      if (!ok) return;
      if (n <= CB) {
        for (int t = tid; t < n * n; t += CNT) {
          const int i = t % n, j = t / n;
          Rinv[(size_t)i + (size_t)j * ldri] = i <= j ? Sc<T>::conj(sm[CB * CLD + j * CLD + i]) : Sc<T>::zero();
        }
      }
    }
    if (rest <= 0) return;
    if (tid == 0) {
      int ok = 1;
      const long long t0 = clock64();
      while (true) {
        unsigned r;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(r) : "l"(&cb->ready) : "memory");
        if ((int)r > kb) break;
        if (*(volatile int*)&cb->bar.abort) { ok = 0; break; }
        if (clock64() - t0 > kBarWait) { atomicExch(&cb->bar.abort, 1); ok = 0; break; }
      }
      if (!ok) atomicOr(&dst->timeout, 32);
      s_ok = ok && !*(volatile int*)&cb->fail;
    }
    __syncthreads();
    if (!s_ok) return;
    // B: block row
    for (int t = tid; t < CB * CB; t += CNT) sm[(t % CB) * CLD + t / CB] = ld_cg(Mk + t);
    __syncthreads();
    T* colb = sm + CB * CLD + warp * CB;
    for (int c = off + b + gw; c < n; c += nw) {
      T* g = G + (size_t)off + (size_t)c * ldg;
      colb[lane] = ld_cg(g + lane);  // (b == CB: there are columns to the right)
      __syncwarp();
      T a = Sc<T>::zero();
#pragma unroll 4
      for (int p = 0; p < CB; ++p) Sc<T>::fma(a, sm[lane * CLD + p], colb[p]);
      g[lane] = a;
      __syncwarp();
    }
    if (!grid_barrier(&cb->bar, G_, bars)) {
      if (tid == 0) atomicOr(&dst->timeout, 32);
      return;
    }
    // C: trailing tiles (tp <= tq)
    const int nt = (rest + CT - 1) / CT, tiles = nt * (nt + 1) / 2, o2 = off + b;
    T* P = sm + (size_t)warp * 2 * CT * CLD;
    T* Q = P + CT * CLD;
    for (int t = gw; t < tiles; t += nw) {
      int tq = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
      while (tq * (tq + 1) / 2 > t) --tq;
      while ((tq + 1) * (tq + 2) / 2 <= t) ++tq;
      const int tp = t - tq * (tq + 1) / 2;
      const int p0 = o2 + tp * CT, q0 = o2 + tq * CT;
#pragma unroll
      for (int c = 0; c < CT; ++c) {
        P[c * CLD + lane] = p0 + c < n ? ld_cg(G + (size_t)(off + lane) + (size_t)(p0 + c) * ldg) : Sc<T>::zero();
        Q[c * CLD + lane] = q0 + c < n ? ld_cg(G + (size_t)(off + lane) + (size_t)(q0 + c) * ldg) : Sc<T>::zero();
      }
      __syncwarp();
      const int p = lane & 7, q = lane >> 3;  // entries (p, q) and (p, q + 4)
      T a0 = Sc<T>::zero(), a1 = Sc<T>::zero();
#pragma unroll 4
      for (int s = 0; s < CB; ++s) {
        const T x = P[p * CLD + s];
        Sc<T>::fmac(a0, x, Q[q * CLD + s]);
        Sc<T>::fmac(a1, x, Q[(q + 4) * CLD + s]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int gp = p0 + p, gq = q0 + q + 4 * h;
        if (gp <= gq && gq < n) {
          T* g = G + (size_t)gp + (size_t)gq * ldg;
          *g = Sc<T>::sub(ld_cg(g), h ? a1 : a0);
        }
      }
      __syncwarp();
    }
    if (!grid_barrier(&cb->bar, G_, bars)) {
      if (tid == 0) atomicOr(&dst->timeout, 32);
      return;
    }
  }
}

// Sum over four lanes, in their order.
__device__ __forceinline__ double quad_sum(double a, int lane) {
  double s = __shfl_sync(0xffffffffu, a, lane & ~3);
#pragma unroll
  for (int o = 1; o < 4; ++o) s += __shfl_sync(0xffffffffu, a, (lane & ~3) + o);
  return s;
}
__device__ __forceinline__ z64 quad_sum(z64 a, int lane) { return z64{quad_sum(a.x, lane), quad_sum(a.y, lane)}; }

// Columns blockIdx.x and n - 1 - blockIdx.x of R^{-1} (n > CB).  The column is all the shared memory
// it takes: 227 KB hold 14528 complex rows.
template <class T>
__global__ void __launch_bounds__(128) trinv_kernel(int n, const T* R, int ldr,
                                                    const T* Mb, T* Rinv, int ldri,
                                                    const DevStatus* dst) {
  dep_wait();
  extern __shared__ __align__(16) unsigned char inv_smem[];
  T* x = (T*)inv_smem;
  if (dst->chol_info) return;
  const int tid = threadIdx.x, lane = tid & 31;
  for (int half = 0; half < 2; ++half) {
    const int j = half ? n - 1 - (int)blockIdx.x : (int)blockIdx.x;
    if (half && j <= (int)blockIdx.x) break;
    const int kj = j / CB, jj = j - kj * CB;
    for (int i = tid; i < kj * CB; i += 128) x[i] = Sc<T>::zero();
    // R_kk^{-1} e_jj: column jj of M^H
    if (tid < CB) x[kj * CB + tid] = tid <= jj ? Sc<T>::conj(Mb[(size_t)kj * CB * CB + jj + tid * CB]) : Sc<T>::zero();
    __syncthreads();
    for (int k = kj; k > 0; --k) {
      const int off = k * CB, len = k == kj ? jj + 1 : CB;
      // rows above the block
      for (int i = tid; i < off; i += 128) {
        T a = x[i];
        const T* r = R + (size_t)i + (size_t)off * ldr;
#pragma unroll 4
        for (int s = 0; s < len; ++s) Sc<T>::fma(a, r[(size_t)s * ldr], Sc<T>::scale(x[off + s], -1.0));
        x[i] = a;
      }
      __syncthreads();
      // block k - 1: x <- R_kk^{-1} x = M^H x, four lanes to a row, each a quarter of its sum
      const T* M = Mb + (size_t)(k - 1) * CB * CB;
      const int row = tid >> 2, part = tid & 3;
      T a = Sc<T>::zero();
#pragma unroll
      for (int p = 8 * part; p < 8 * part + 8; ++p) Sc<T>::fmac(a, M[p + row * CB], x[off - CB + p]);
      a = quad_sum(a, lane);
      __syncthreads();
      if (part == 0) x[off - CB + row] = a;
      __syncthreads();
    }
    for (int i = tid; i < n; i += 128) Rinv[(size_t)i + (size_t)j * ldri] = i <= j ? x[i] : Sc<T>::zero();
    __syncthreads();
  }
}

}  // namespace

size_t chol_work_bytes(int n, size_t elem) { return sizeof(CholBar) + 256 + elem * CB * CB * (size_t)ceil_div(n, CB); }

template <class T>
int chol_inverse(cudaStream_t st, int n, T* G, int ldg, double shift_factor, T* Rinv, int ldri, Scratch work,
                 DevStatus* dst, int* launches) {
  if (n <= 0) return 0;
  if (work.bytes < chol_work_bytes(n, sizeof(T))) return CHASE_ERR_OOM;
  CholBar* cb = (CholBar*)work.ptr;
  T* Mb = (T*)((char*)work.ptr + 256);
  // CTAs: eight tiles of the first trailing update per warp, at most one per SM
  const long long nt = ceil_div(std::max(0, n - CB), CT), tiles = nt * (nt + 1) / 2;
  int grid = (int)std::max(1LL, std::min<long long>(kNumSMs, (tiles + CW - 1) / CW));
  const int smem = (int)sizeof(T) * std::max(CW * 2 * CT * CLD, 2 * CB * CLD);
  CHASE_CUDA_TRY(cudaFuncSetAttribute(chol_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  CHASE_CUDA_TRY(cudaMemsetAsync(cb, 0, sizeof(CholBar), st));
  void* args[] = {(void*)&n, (void*)&G, (void*)&ldg, (void*)&shift_factor, (void*)&Mb, (void*)&Rinv,
                  (void*)&ldri, (void*)&cb, (void*)&dst};
  CHASE_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)chol_kernel<T>, dim3(grid), dim3(CNT), args, (size_t)smem, st));
  if (launches) ++*launches;
  if (n > CB) {
    const size_t xs = sizeof(T) * (size_t)ceil_div(n, CB) * CB;
    // (always the same value: another thread may be about to launch with a longer column)
    CHASE_CUDA_TRY(cudaFuncSetAttribute(trinv_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax));
    launch_dep(st, ceil_div(n, 2), 128, xs, trinv_kernel<T>, n, G, ldg, Mb, Rinv, ldri, dst);
    if (launches) ++*launches;
  }
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

template int chol_inverse<double>(cudaStream_t, int, double*, int, double, double*, int, Scratch, DevStatus*, int*);
template int chol_inverse<z64>(cudaStream_t, int, z64*, int, double, z64*, int, Scratch, DevStatus*, int*);

}  // namespace chase
