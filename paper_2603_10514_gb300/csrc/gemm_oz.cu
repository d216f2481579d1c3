// gemm_oz.cu -- FP64-accurate dense products on the BF16 tensor cores by the
// Ozaki scheme II (Ozaki, Uchino & Imamura, "Ozaki Scheme II: A GEMM-oriented
// emulation of floating-point matrix multiplication using an integer modular
// technique", 2025): the filter's A*V, the Rayleigh-Ritz product A*Q and the
// block products of the QR and Rayleigh-Ritz steps.
//
// Integer operands.  Every row m of the (stacked real) left operand is scaled by
// 2^{57 - e_m} (max_k |L[m,k]| < 2^{e_m}) and every column c of the right
// operand by 2^{57 - f_c}; each scaled entry is rounded to the nearest integer,
// so |L_int|, |V_int| <= 2^57 and the rounding error is at most 2^-58 of the
// row (column) scale.  The product of the integer matrices
//   X[m, c] = sum_k L_int[m, k] V_int[k, c],   |X| <= K 2^114,
// is computed EXACTLY, and (A V)[m, c] = 2^{e_m + f_c - 114} X[m, c] is then
// within K 2^-57 max_k|L[m,k]| max_k|V[k,c]| of the exact product: the accuracy
// class of an FP64 GEMM.
//
// Exact integer product by the Chinese remainder theorem.  With S = 17 pairwise
// coprime moduli p_j <= 256 (product P ~ 2^132.95 > 2 K 2^114 for K <= 2^17),
// X is recovered from its residues X mod p_j.  Each residue needs one product
// of residue matrices: L_int mod p_j and V_int mod p_j are stored in symmetric
// range (|r| <= 128, exact in BF16), so one BF16 tensor-core product per
// modulus forms sum_k (L mod p)(V mod p), whose partial sums over a K chunk of
// 1024 stay within 1024 * 128^2 = 2^24 and are therefore exact in the tensor
// core's FP32 accumulator; the epilogue adds the chunks as 32-bit integers and
// reduces mod p_j at the end.  17 BF16 products replace the FP64 product.
// Reconstruction (crt_finish): X = sum_j r_j C_j mod P with C_j = (P/p_j) *
// ((P/p_j)^{-1} mod p_j), in 160-bit integer arithmetic (32-bit limbs), mapped
// to the symmetric range (-P/2, P/2] and rounded once to FP64.
//
// Complex A*V and A*Q products use a second set of moduli in which -1 is a square (every prime
// factor is 1 mod 4): Z_p[i] then splits into two copies of Z_p, and one complex product takes
// TWO real modular products per modulus (see "Complex products in split residue rings").
//
// Modular product kernel (ozm_kernel): CTA pairs (clusters of two along grid x), one pair
// per (256-row block, column tile of BN <= 320 columns, modulus[, K split]).  The even CTA
// issues tcgen05.mma.cta_group::2.kind::f16 (M 256, N <= 160, K 16) over the pair: each CTA
// holds its own 128 rows of A and half of each MMA's V rows in shared memory, and its 128 rows of
// the accumulators in its own TMEM.  Tiles above 160 columns are two halves with an MMA each on
// the same A block.
// What binds is the operand feed: a stage's copies must land within the time the other stages'
// MMAs take (DRAM and L2 latency), and every SM takes at most ~67 bytes per clock from L2.  The
// wide tile moves 59 bytes per clock of MMA time (128 rows of A and 152 of V per 304 columns; 71
// for 208 columns), and a 64-wide K block of it still holds 8 MMAs, the fewest that hide a
// barrier round trip between producer and issuer, so six stages fit where three K-128 stages of
// a 256-column tile did.
// The halves' exact K chunks are staggered by half a chunk over THREE accumulators of 160
// columns: while one half's finished chunk is read out, the other half and the next chunk go
// on in the other two.  16 epilogue warps read TMEM with tcgen05.ld; their sums take 80
// registers, which setmaxnreg moves over from the producer's warpgroup.  The issuing warp's
// loop is warp-uniform (one lane's instructions are predicated): under a lane-0 branch every
// MMA took ~100 cycles to issue, which bound every tile narrower than 256 columns.
// Measured against two 256-column accumulators, K-128 stages and a lane-0 issuer (full-size
// modular products, real data): 600 columns complex 2616 -> 2159 us (1.68 PFLOP/s; cuBLAS holds
// 1.73 under the power cap), real 1427 -> 1100 us; one tile of 64-256 columns stays bound by the
// stream of A's planes from HBM (941 us at 64 columns, 6.4 TB/s).
// All mbarrier waits are bounded; on expiry the kernel records the failure in
// the device status word, waits (bounded) for its copies and MMAs in flight,
// frees its TMEM and returns.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <type_traits>

#include "../../include/chase_gb300.h"
#include "common.cuh"
#include "kernels.h"
#include "tcgen05.cuh"

namespace chase {

#define TRY_OZ(x)          \
  do {                     \
    int _rc = (x);         \
    if (_rc) return _rc;   \
  } while (0)

namespace {

// ---------------------------------------------------------------------------
// Moduli and CRT constants (computed at compile time)
// ---------------------------------------------------------------------------
constexpr int OZ_KBITS = 57;  // integer operands: |x_int| <= 2^57
// 17 pairwise coprime moduli <= 256 (256 = 2^8; 255 = 3 5 17; 253 = 11 23; 247 = 13 19;
// 217 = 7 31; the others prime): P = prod p_j ~ 2^132.95 > 2 * 2^17 * 2^114.
__host__ __device__ constexpr int oz_modulus(int j) {
  constexpr int t[kOzModuli] = {256, 255, 253, 251, 247, 241, 239, 233, 229,
                                227, 223, 217, 211, 199, 197, 193, 191};
  return t[j];
}
static_assert(kOzPlaneBytes == 2 * kOzModuli, "workspace plane size");
static_assert(kOzMaxK <= (1 << 17), "K bound of the modulus product");

struct Big {  // unsigned 160-bit integer, little-endian 32-bit limbs
  uint32_t w[5];
};

constexpr Big big_small(uint32_t x) { return Big{{x, 0, 0, 0, 0}}; }
constexpr Big big_mul_small(Big a, uint32_t k) {
  uint64_t c = 0;
  for (int i = 0; i < 5; ++i) {
    const uint64_t t = (uint64_t)a.w[i] * k + c;
    a.w[i] = (uint32_t)t;
    c = t >> 32;
  }
  return a;
}
constexpr uint32_t big_mod_small(Big a, uint32_t p) {
  uint64_t r = 0;
  for (int i = 4; i >= 0; --i) r = ((r << 32) | a.w[i]) % p;
  return (uint32_t)r;
}
constexpr uint32_t inv_mod(uint32_t a, uint32_t p) {  // a^{-1} mod p, gcd(a, p) = 1
  long long t = 0, nt = 1, r = p, nr = a % p;
  while (nr != 0) {
    const long long q = r / nr;
    long long tmp = t - q * nt; t = nt; nt = tmp;
    tmp = r - q * nr; r = nr; nr = tmp;
  }
  return (uint32_t)(t < 0 ? t + p : t);
}

struct CrtTable {
  int p[kOzModuli];          // the moduli
  uint32_t C[kOzModuli][5];  // C_j = (P / p_j) ((P / p_j)^{-1} mod p_j) < P
  uint32_t P[5];
  float p96_over_P;          // 2^96 / P (rounded)
};

constexpr CrtTable make_crt_table() {
  CrtTable t{};
  Big P = big_small(1);
  for (int j = 0; j < kOzModuli; ++j) {
    t.p[j] = oz_modulus(j);
    P = big_mul_small(P, (uint32_t)oz_modulus(j));
  }
  for (int j = 0; j < kOzModuli; ++j) {
    Big Mj = big_small(1);
    for (int i = 0; i < kOzModuli; ++i)
      if (i != j) Mj = big_mul_small(Mj, (uint32_t)oz_modulus(i));
    const uint32_t inv = inv_mod(big_mod_small(Mj, (uint32_t)oz_modulus(j)), (uint32_t)oz_modulus(j));
    const Big Cj = big_mul_small(Mj, inv);
    for (int l = 0; l < 5; ++l) t.C[j][l] = Cj.w[l];
  }
  double pd = 0.0;
  for (int l = 4; l >= 0; --l) {
    t.P[l] = P.w[l];
    pd = pd * 4294967296.0 + (double)P.w[l];
  }
  t.p96_over_P = (float)(79228162514264337593543950336.0 / pd);  // 2^96 / P
  return t;
}

__constant__ CrtTable c_crt = make_crt_table();

// Compile-time checks of the number theory the reconstruction relies on: the moduli are
// pairwise coprime, C_j is 1 mod p_j and 0 mod every other modulus, and P exceeds twice the
// largest integer product, 2 * 2^17 * 2^114 = 2^132 (limb 4 holds P / 2^128).
constexpr int oz_gcd(int a, int b) { return b == 0 ? a : oz_gcd(b, a % b); }
constexpr bool oz_moduli_coprime() {
  for (int i = 0; i < kOzModuli; ++i)
    for (int j = i + 1; j < kOzModuli; ++j)
      if (oz_gcd(oz_modulus(i), oz_modulus(j)) != 1) return false;
  return true;
}
constexpr bool oz_crt_basis_ok() {
  const CrtTable t = make_crt_table();
  for (int j = 0; j < kOzModuli; ++j) {
    const Big Cj{{t.C[j][0], t.C[j][1], t.C[j][2], t.C[j][3], t.C[j][4]}};
    for (int i = 0; i < kOzModuli; ++i)
      if (big_mod_small(Cj, (uint32_t)oz_modulus(i)) != (i == j ? 1u : 0u)) return false;
  }
  return true;
}
static_assert(oz_moduli_coprime(), "moduli must be pairwise coprime");
static_assert(oz_crt_basis_ok(), "CRT basis: C_j = 1 mod p_j, 0 mod p_i");
static_assert(make_crt_table().P[4] >= (1u << (2 * OZ_KBITS + 17 + 1 - 128)), "P > 2 K 2^114");
// The modular epilogue reduces a split's sum |s| <= kOzSplitMaxK * 128^2 = 2^30 with the
// float quotient q = floor(fl(fl(s) * fl(1/p))): fl(s) is within 32 of s and the two roundings
// add a relative 2^-23, so q is within 32/p + 2^30 2^-23 / p < 1 of s/p for p > 160 and one
// correction step lands in [0, p).
constexpr bool oz_moduli_above(int lo) {
  for (int j = 0; j < kOzModuli; ++j)
    if (oz_modulus(j) <= lo) return false;
  return true;
}
static_assert(oz_moduli_above(160), "epilogue reduction: p > 160");
static_assert((long long)kOzSplitMaxK * 128 * 128 <= (1ll << 30), "epilogue reduction: |sum| <= 2^30");
static_assert(kOzMaxK <= kOzMaxSplits * kOzSplitMaxK, "every admissible K fits the splits");

// ---------------------------------------------------------------------------
// Complex products in split residue rings
// ---------------------------------------------------------------------------
// For a modulus p whose prime factors are all 1 mod 4 there is an s with s^2 = -1 mod p, and
//   a + i b  ->  (a + s b, a - s b) mod p
// turns a complex product into two independent real ones:  with U = sum (Ar + s Ai)(Vr + s Vi)
// and W = sum (Ar - s Ai)(Vr - s Vi),  Re(A V) = (U + W) / 2  and  Im(A V) = (U - W) / (2 s)
// mod p.  Two modular products per modulus where the product of order n by Gauss's form takes
// three and the stacked real operator of order 2n four; the integers of A and V, and so the
// results, are the same bit for bit.  Moduli up to 509 keep residues |r| <= 254 exact in BF16
// (8 significant bits) and give ~8.8 bits each: 15 of them (P ~ 2^131.4) cover |Re|, |Im| <=
// 2 K 2^114 for K <= 2^15, 16 (2^139.8) every admissible K.  Their price: an exact FP32 chunk
// is 256 wide (256 254^2 < 2^24) instead of 1024, and a residue of the product takes two bytes.
// Per complex product of order n: 30 BF16 products (17 moduli x 3 by Gauss's form: 51).
// Bound: the tensor pipe and its L2 feed.  Measured (filter call, degrees 10-36, GB300): n = 10000,
// 600 columns 136.0 -> 84.0 ms, n = 3000, 180 columns 11.50 -> 7.06 ms against Gauss's form.
__host__ __device__ constexpr int ring_modulus(int j) {
  constexpr int tr[kRingModuli] = {509, 505, 493, 481, 461, 457, 449, 433,
                                   421, 409, 401, 397, 389, 373, 353, 349};
  return tr[j];
}
// s with s^2 = -1 mod p_j
__host__ __device__ constexpr uint32_t ring_root(int j) {
  const uint32_t p = (uint32_t)ring_modulus(j);
  for (uint32_t s = 1; s < p; ++s)
    if ((s * s + 1) % p == 0) return s;
  return 0;
}

// CRT constants of the first NM ring moduli: X_re = sum_j (U_j + W_j) Cre_j mod P and
// X_im = sum_j (U_j - W_j + p_j) Cim_j mod P, with Cre_j = 1/2 and Cim_j = 1/(2 s_j) mod p_j,
// both 0 mod every other modulus.
template <int NM>
struct RingTable {
  uint32_t Cre[NM][5], Cim[NM][5];
  uint32_t P[5];
  float p96_over_P;
};

template <int NM>
constexpr RingTable<NM> make_ring_table() {
  RingTable<NM> t{};
  Big P = big_small(1);
  for (int j = 0; j < NM; ++j) P = big_mul_small(P, (uint32_t)ring_modulus(j));
  for (int j = 0; j < NM; ++j) {
    const uint32_t p = (uint32_t)ring_modulus(j);
    Big Mj = big_small(1);
    for (int i = 0; i < NM; ++i)
      if (i != j) Mj = big_mul_small(Mj, (uint32_t)ring_modulus(i));
    const uint32_t inv = inv_mod(big_mod_small(Mj, p), p);
    const Big Cre = big_mul_small(Mj, inv * inv_mod(2, p) % p);
    const Big Cim = big_mul_small(Mj, inv * inv_mod(2 * ring_root(j) % p, p) % p);
    for (int l = 0; l < 5; ++l) {
      t.Cre[j][l] = Cre.w[l];
      t.Cim[j][l] = Cim.w[l];
    }
  }
  double pd = 0.0;
  for (int l = 4; l >= 0; --l) {
    t.P[l] = P.w[l];
    pd = pd * 4294967296.0 + (double)P.w[l];
  }
  t.p96_over_P = (float)(79228162514264337593543950336.0 / pd);
  return t;
}
constexpr int kRingShort = 15;
__constant__ RingTable<kRingShort> c_ring15 = make_ring_table<kRingShort>();
__constant__ RingTable<kRingModuli> c_ring16 = make_ring_table<kRingModuli>();
template <int NM> __device__ __forceinline__ const RingTable<NM>& ring_table();
template <> __device__ __forceinline__ const RingTable<kRingShort>& ring_table<kRingShort>() { return c_ring15; }
template <> __device__ __forceinline__ const RingTable<kRingModuli>& ring_table<kRingModuli>() { return c_ring16; }

constexpr bool ring_moduli_ok() {
  for (int i = 0; i < kRingModuli; ++i) {
    const uint32_t p = (uint32_t)ring_modulus(i), s = ring_root(i);
    if (s == 0 || (s * s + 1) % p != 0) return false;
    // exact chunks, with the folded sum of the earlier ones (fold2)
    if (kRingChunk * (long long)(p / 2) * (p / 2) + p >= (1ll << 24)) return false;
    for (int j = i + 1; j < kRingModuli; ++j)
      if (oz_gcd((int)p, ring_modulus(j)) != 1) return false;
  }
  return true;
}
template <int NM>
constexpr bool ring_crt_ok() {
  const RingTable<NM> t = make_ring_table<NM>();
  for (int j = 0; j < NM; ++j) {
    const Big Cre{{t.Cre[j][0], t.Cre[j][1], t.Cre[j][2], t.Cre[j][3], t.Cre[j][4]}};
    const Big Cim{{t.Cim[j][0], t.Cim[j][1], t.Cim[j][2], t.Cim[j][3], t.Cim[j][4]}};
    for (int i = 0; i < NM; ++i) {
      const uint32_t p = (uint32_t)ring_modulus(i);
      if (big_mod_small(Cre, p) * 2 % p != (i == j ? 1u : 0u)) return false;
      if (big_mod_small(Cim, p) * (2 * ring_root(i) % p) % p != (i == j ? 1u : 0u)) return false;
    }
  }
  return true;
}
static_assert(ring_moduli_ok(), "ring moduli: -1 a square, exact chunks, pairwise coprime");
static_assert(ring_crt_ok<kRingShort>() && ring_crt_ok<kRingModuli>(), "ring CRT basis");
// P > 2 * (2 K 2^114): K <= 2^15 with 15 moduli, K <= 2^17 with 16
static_assert(make_ring_table<kRingShort>().P[4] >= (1u << (2 * OZ_KBITS + 15 + 2 - 128)), "ring range, 15");
static_assert(make_ring_table<kRingModuli>().P[4] >= (1u << (2 * OZ_KBITS + 17 + 2 - 128)), "ring range, 16");
static_assert(kRingShortMaxK == (1 << 15), "ring_moduli()");

__constant__ int c_ring_p[kRingModuli] = {ring_modulus(0),  ring_modulus(1),  ring_modulus(2),
                                          ring_modulus(3),  ring_modulus(4),  ring_modulus(5),
                                          ring_modulus(6),  ring_modulus(7),  ring_modulus(8),
                                          ring_modulus(9),  ring_modulus(10), ring_modulus(11),
                                          ring_modulus(12), ring_modulus(13), ring_modulus(14),
                                          ring_modulus(15)};

constexpr int MBM = 128, MBK = 64;
constexpr int MH_MAX = 160;         // columns of one MMA (one accumulator)
constexpr int MBN_MAX = 2 * MH_MAX;
constexpr int MNST_MAX = 8;
constexpr int M_EPI_WARPS = 16;
constexpr int M_THREADS = 128 + 32 * M_EPI_WARPS;  // a warpgroup for producer and issuer
constexpr int M_REG_MAIN = 64, M_REG_EPI = 104;    // of 5 x 96 registers at launch
static_assert(M_REG_MAIN + 4 * M_REG_EPI <= 5 * 96, "register split");
constexpr int M_CHUNK = 1024 / MBK;                // K blocks of an exact chunk
constexpr int M_A1 = MBM * MBK * 2;                // 16 KB: 128 rows of A, one K block
constexpr int M_STAGES = 6 * (M_A1 + MH_MAX * MBK * 2);  // bytes for stages: six of the widest tile
constexpr int M_SMEM = M_STAGES + 1024 + 256;
constexpr uint32_t M_TMEM_COLS = 512;              // three accumulators of 160 columns
static_assert(M_SMEM <= 232448, "shared memory");
static_assert(M_A1 % 1024 == 0, "stage alignment (128-byte swizzle atoms)");
// K blocks whose products of residues mod p_j, with the folded sum of the earlier ones (fold2),
// stay exact integers below 2^24: 4 for 509 to 8 for 349
__host__ __device__ constexpr int ring_chunk_of(int j) {
  const int h = ring_modulus(j) / 2;
  return ((1 << 24) - 1 - 2 * h) / (h * h) / MBK;
}
static_assert(ring_chunk_of(0) * MBK == kRingChunk, "shortest exact chunk");
__constant__ int c_ring_chunk[kRingModuli] = {ring_chunk_of(0),  ring_chunk_of(1),  ring_chunk_of(2),
                                              ring_chunk_of(3),  ring_chunk_of(4),  ring_chunk_of(5),
                                              ring_chunk_of(6),  ring_chunk_of(7),  ring_chunk_of(8),
                                              ring_chunk_of(9),  ring_chunk_of(10), ring_chunk_of(11),
                                              ring_chunk_of(12), ring_chunk_of(13), ring_chunk_of(14),
                                              ring_chunk_of(15)};
__device__ __forceinline__ int ring_chunk(int j) { return c_ring_chunk[j]; }

// Shape of a column tile of BN columns (a multiple of 16): one or two halves (multiples of 16),
// K blocks per stage (8 MMAs where BN > 64 needs them), bytes of a stage and stages that fit.
struct TileShape {
  int h0, h1, ks, hb, stage, nst;
};
__host__ __device__ inline TileShape tile_shape(int BN) {
  TileShape s;
  s.h0 = BN <= MH_MAX ? BN : (BN / 2 + 15) / 16 * 16;
  s.h1 = BN - s.h0;
  s.ks = s.h1 ? 1 : 2;
  s.hb = (s.h0 / 2) * MBK * 2;  // bytes of one CTA's V rows of a half (the box of the V map)
  s.stage = s.ks * (M_A1 + (s.h1 ? 2 : 1) * s.hb);
  s.nst = M_STAGES / s.stage < MNST_MAX ? M_STAGES / s.stage : MNST_MAX;
  return s;
}
using namespace tc;

// ---------------------------------------------------------------------------
// Modular products: R[z][c][r] = (sum_{k in split} Lres_j[r, k] Vres_j[k, c]) mod p_j,
// z = split * S + j (grid z).  Lres planes row-major (rows x kp), Vres planes column-major
// (kp x ncols); both K-padded with zeros to kp (a multiple of 64).
// ---------------------------------------------------------------------------
// s mod p in [0, p) by a float quotient that is off by at most one.
__device__ __forceinline__ int mod_sum(int s, int p, float ip) {
  const int q = (int)floorf((float)s * ip);
  int r = s - q * p;
  if (r < 0) r += p;
  if (r >= p) r -= p;
  return r;
}

__device__ __forceinline__ uint64_t pack2(float x, float y) {
  return (uint64_t)__float_as_uint(x) | ((uint64_t)__float_as_uint(y) << 32);
}
// Two sums mod p advanced by one chunk each: s = acc + v is an exact integer below 2^24
// (256 254^2 + p/2), q = round(s / p) to within 2^-8, and s - q p, exact, lies within 0.51 p.
// Four packed FP32 operations per pair: float-to-integer conversions issue at 16 per clock
// per SM and would take longer than the chunk's MMAs.
__device__ __forceinline__ uint64_t fold2(uint64_t acc, uint32_t v0, uint32_t v1, uint64_t ip2, uint64_t np2) {
  const uint64_t magic = 0x4B4000004B400000ull;   // 1.5 * 2^23, twice
  uint64_t v, s, q, r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "r"(v0), "r"(v1));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(s) : "l"(acc), "l"(v));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(q) : "l"(s), "l"(ip2), "l"(magic));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(q) : "l"(q), "l"(magic));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(q), "l"(np2), "l"(s));
  return r;
}

// One CTA of a pair (clusters of two CTAs along grid x): this CTA's rows [m0, m0 + 128)
// and the pair's columns [n0, n0 + BN) of modulus jm over the K blocks [kbeg, kbeg + nkb);
// residues into Rv (column-major M x N).  A stage may hold one block past the last (zero-filled
// beyond kp, else the next split's): it is copied but not multiplied.
// RING: modulus jm of the ring set, 256-wide exact chunks folded mod p as they come (no limit
// on the length of K), two-byte residues.
//
// Accumulators: at switch s = 1, 2, ... (every half chunk; one-half tiles: every chunk) one
// half's finished accumulator goes to the epilogue and the half moves on to the accumulator
// that the switch before gave up.  Two halves: odd switches are half 1's, even ones half 0's;
// accumulator (2 - s) mod 3 is given up for (3 - s) mod 3.  One half: (s - 1) & 1 for s & 1.
// After the last block every half's accumulator follows in the same order.
template <bool RING>
__device__ __forceinline__ void ozm_pair_tile(const CUtensorMap* mapA, const CUtensorMap* mapV,
                                              int M, int N, int BN, int col0, int m0, int n0,
                                              int jm, int kbeg, int nkb, void* __restrict__ Rv,
                                              DevStatus* status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = (uint64_t*)(smem + M_STAGES);
  uint64_t* full = bars;                    // [MNST_MAX] stage loaded (both CTAs' copies; the even CTA's)
  uint64_t* empty = bars + MNST_MAX;        // [MNST_MAX] stage read by the pair's MMAs
  uint64_t* cfull = bars + 2 * MNST_MAX;    // [3] accumulator b holds a finished chunk
  uint64_t* cfree = cfull + 3;              // [3] accumulator b read out by both CTAs (the even CTA's)
  uint64_t* tdone = cfree + 3;              // every MMA finished
  uint32_t* tslot = (uint32_t*)(tdone + 1);
  int* s_err = (int*)(tslot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const TileShape ts = tile_shape(BN);
  const bool two = ts.h1 > 0;
  const int nst = (nkb + ts.ks - 1) / ts.ks;
  const int chunk = RING ? ring_chunk(jm) : M_CHUNK;  // K blocks of an exact chunk
  const int gap1 = two ? chunk / 2 : chunk, gap0 = two ? chunk - gap1 : chunk;  // blocks before odd / even switches
  const int nsw = (two ? 2 : 1) * ((nkb - 1) / chunk) + (two && (nkb - 1) % chunk >= gap1 ? 1 : 0);  // switches
  const int ndrain = nkb > 0 ? nsw + (two ? 2 : 1) : 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < MNST_MAX; ++i) { bar_init(&full[i], 1); bar_init(&empty[i], 1); }
    for (int b = 0; b < 3; ++b) { bar_init(&cfull[b], 1); bar_init(&cfree[b], 2 * M_EPI_WARPS); }
    bar_init(tdone, 1);
    *s_err = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {  // one warp of each CTA of the pair allocates the pair's accumulators
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(s32(tslot)),
                 "r"(M_TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync();  // both CTAs' barriers initialised before any copy or arrival crosses over
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  // (the set-up above runs beside the end of the launch before; the reconstruction after it is not
  // placed early, on the few SMs that the last tiles leave free: n = 1000 real, 30 columns, a filter
  // of 20 steps 492 -> 444 us, a solve 9.1 -> 8.1 ms)
  dep_wait(false);

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(M_REG_MAIN));
    if (warp == 0 && lane == 0) {
      // ---------------- producer (both CTAs): own A rows, own half of each V half tile ----------------
      const uint32_t bytes = (uint32_t)(2 * ts.stage);  // the pair's copies of a stage
      const uint32_t full0 = peer_addr(full, 0);
      const int v0 = col0 + n0 + (int)rank * (ts.h0 >> 1), v1 = col0 + n0 + ts.h0 + (int)rank * (ts.h1 >> 1);
      int issued = 0, s = 0;
      uint32_t ph = 1;
      for (int it = 0; it < nst && !*(volatile int*)s_err; ++it) {
        if (!bar_wait(&empty[s], ph)) { atomicOr(s_err, 1); break; }
        if (rank == 0) bar_expect(&full[s], bytes);
        unsigned char* st = smem + s * ts.stage;
        const uint32_t fb = full0 + 8u * (uint32_t)s;
        const int x = (kbeg + it * ts.ks) * MBK;
        tma3_pair(st, mapA, fb, x, m0, jm);
        if (two) {
          tma3_pair(st + M_A1, mapV, fb, x, v0, jm);
          tma3_pair(st + M_A1 + ts.hb, mapV, fb, x, v1, jm);
        } else {
          tma3_pair(st + M_A1, mapA, fb, x + MBK, m0, jm);
          tma3_pair(st + 2 * M_A1, mapV, fb, x, v0, jm);
          tma3_pair(st + 2 * M_A1 + ts.hb, mapV, fb, x + MBK, v0, jm);
        }
        issued = it + 1;
        if (++s == ts.nst) { s = 0; ph ^= 1; }
      }
      // every release of this CTA's stages has arrived (no arrival may reach it after exit) ...
      for (int it = issued; it < issued + ts.nst; ++it)
        if (!bar_wait(&empty[it % ts.nst], (uint32_t)(((it / ts.nst) & 1) ^ 1))) { atomicOr(s_err, 1); break; }
      // ... and, in the even CTA, every copy of both CTAs has landed
      if (rank == 0)
        for (int b = max(0, issued - ts.nst); b < issued; ++b)
          if (!bar_wait(&full[b % ts.nst], (uint32_t)((b / ts.nst) & 1))) { atomicOr(s_err, 1); break; }
    } else if (warp == 1 && rank == 0) {
      // ---------------- MMA issuer (even CTA, the whole warp): M 256 x N h x K 16 over the pair ----------------
      const uint32_t leader = elect_lane();
      const uint32_t id = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * MBM) >> 4) << 24);
      const uint32_t id0 = id | ((uint32_t)(ts.h0 >> 3) << 17), id1 = id | ((uint32_t)(ts.h1 >> 3) << 17);
      uint32_t d0 = tmem, d1 = tmem + MH_MAX;  // the halves' accumulators
      uint32_t acc0 = 0, acc1 = 0;             // 0: the next MMA starts a chunk
      uint32_t given = 0, fph = 0;             // accumulators given up before, phases of their release
      int sw = 0, left = gap1;                 // switches made, blocks to the next one
      bool bad = false;
      int s = 0;
      uint32_t ph = 0;
      for (int it = 0; it < nst && !bad; ++it) {
        if (!bar_poll(&full[s], ph)) { bad = true; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t sa = s32(smem + s * ts.stage);
        for (int u = 0; u < ts.ks; ++u) {
          if (it * ts.ks + u >= nkb) break;
          if (left == 0) {
            ++sw;
            left = (sw & 1) ? gap0 : gap1;
            const int from = two ? (sw % 3 == 0 ? 2 : 2 - sw % 3) : (sw - 1) & 1;
            const int to = two ? (sw % 3 == 0 ? 0 : 3 - sw % 3) : sw & 1;
            commit_pair(&cfull[from], leader);
            if ((given >> to) & 1) {  // read out since it was given up
              if (!bar_poll_cluster(&cfree[to], (fph >> to) & 1)) { bad = true; break; }
              // the stage's fence was before this wait: the MMAs below overwrite what was read out
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              fph ^= 1u << to;
            }
            given |= 1u << from;
            if (two && (sw & 1)) { d1 = tmem + (uint32_t)to * MH_MAX; acc1 = 0; }
            else { d0 = tmem + (uint32_t)to * MH_MAX; acc0 = 0; }
          }
          --left;
          const uint64_t da = desc_sw128(sa + u * M_A1);
          const uint64_t dv = desc_sw128(sa + ts.ks * M_A1 + u * ts.hb);
#pragma unroll
          for (int k = 0; k < MBK / 16; ++k) {
            mma_pair(d0, da + 2 * k, dv + 2 * k, id0, acc0, leader);
            acc0 = 1;
          }
          if (two) {
            const uint64_t dw = desc_sw128(sa + M_A1 + ts.hb);
#pragma unroll
            for (int k = 0; k < MBK / 16; ++k) {
              mma_pair(d1, da + 2 * k, dw + 2 * k, id1, acc1, leader);
              acc1 = 1;
            }
          }
        }
        if (bad) break;
        commit_pair(&empty[s], leader);
        if (++s == ts.nst) { s = 0; ph ^= 1; }
      }
      if (bad && lane == 0) atomicOr(s_err, 2);
      // the halves' last chunks, in switch order
      for (int e = nsw + 1; e <= ndrain && !bad; ++e)
        commit_pair(&cfull[two ? (e % 3 == 0 ? 2 : 2 - e % 3) : (e - 1) & 1], leader);
      commit_pair(tdone, leader);
    }
  } else {
    // ---------------- epilogue (both CTAs, own TMEM lanes = own 128 rows) ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(M_REG_EPI));
    // warp w reads TMEM lanes 32 (w % 4) .. +31 (the hardware's lane quarter of the warp) and
    // the quarter (w - 4) / 4 of each half's columns (<= 40)
    const int q = warp & 3, cq = (warp - 4) >> 2;
    const int r = m0 + 32 * q + lane;
    const int cw0 = ts.h0 >> 2, cw1 = ts.h1 >> 2;
    const uint32_t cfree0 = peer_addr(cfree, 0);
    const int pm = RING ? c_ring_p[jm] : c_crt.p[jm];
    const float ip = 1.0f / (float)pm;
    // sums of the chunks: 32-bit integers, or (ring) pairs of floats in (-0.51 p, 0.51 p)
    constexpr int CW = MH_MAX / 4;
    int sum[2][RING ? 1 : CW];
    uint64_t acc[2][RING ? CW / 2 : 1];
    const uint64_t ip2 = pack2(ip, ip), np2 = pack2(-(float)pm, -(float)pm);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
#pragma unroll
      for (int j = 0; j < (RING ? 1 : CW); ++j) sum[h][j] = 0;
#pragma unroll
      for (int j = 0; j < (RING ? CW / 2 : 1); ++j) acc[h][j] = 0;
    }
    uint32_t uses = 0;  // phases of the accumulators' cfull
    bool ok = true;
    auto drain = [&](auto half, int e, int b) {
      constexpr int H = decltype(half)::value;
      const int cw = H ? cw1 : cw0;
      if (!__all_sync(0xffffffffu, bar_wait(&cfull[b], (uses >> b) & 1))) {
        ok = false;
        if (lane == 0) atomicOr(s_err, 4);
        return;
      }
      uses ^= 1u << b;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(b * MH_MAX + cq * cw);
      // eight columns at a time: wider reads spill, and a spill in this loop costs more
#pragma unroll
      for (int g = 0; g < CW / 8; ++g) {
        if (8 * g >= cw) break;
        uint32_t v[8];
        ld8(ta + 8 * g, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if constexpr (RING) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            acc[H][4 * g + j] = fold2(acc[H][4 * g + j], v[2 * j], v[2 * j + 1], ip2, np2);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) sum[H][8 * g + j] += __float2int_rn(__uint_as_float(v[j]));
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0 && e <= nsw) arrive_remote(cfree0 + 8u * (uint32_t)b);
    };
    for (int e = 1; e <= ndrain && ok; ++e) {
      if (!two) drain(std::integral_constant<int, 0>(), e, (e - 1) & 1);
      else if (e & 1) drain(std::integral_constant<int, 1>(), e, e % 3 == 0 ? 2 : 2 - e % 3);
      else drain(std::integral_constant<int, 0>(), e, e % 3 == 0 ? 2 : 2 - e % 3);
    }
    if (__shfl_sync(0xffffffffu, (int)(ok && !*(volatile int*)s_err), 0) && r < M) {
      // the sums mod p in [0, p)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int cw = h ? cw1 : cw0, c0 = n0 + h * ts.h0 + cq * cw;
#pragma unroll
        for (int j = 0; j < CW; ++j) {
          if (j < cw && c0 + j < N) {
            const size_t at = (size_t)(c0 + j) * M + r;
            if constexpr (RING) {
              const int rr = (int)__uint_as_float((uint32_t)(acc[h][j >> 1] >> (32 * (j & 1))));
              ((uint16_t*)Rv)[at] = (uint16_t)(rr < 0 ? rr + pm : rr);
            } else {
              ((uint8_t*)Rv)[at] = (uint8_t)mod_sum(sum[h][j], pm, ip);
            }
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1 && !bar_wait(tdone, 0u) && lane == 0) atomicOr(s_err, 8);
  cluster_sync();  // neither CTA frees the pair's TMEM or exits while the other may signal it
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(M_TMEM_COLS));
  }
  if (threadIdx.x == 32 && *s_err) atomicOr(&status->timeout, *s_err);
}

// Pair index p = blockIdx.x / 2 runs over (row pair, column tile) with the column tiles
// fastest, so the tiles of one row pair read its A rows from L2 at about the same time.
__device__ __forceinline__ void pair_tile_coords(int x, int ntile, int BN, int* m0, int* n0) {
  const int pr = x >> 1;
  *n0 = (pr % ntile) * BN;
  *m0 = (2 * (pr / ntile) + (x & 1)) * MBM;
}

__global__ void __launch_bounds__(M_THREADS, 1)
    ozm_kernel(const __grid_constant__ CUtensorMap mapA, const __grid_constant__ CUtensorMap mapV,
               int M, int N, int BN, int ntile, int col0, int nkb_total, int kbs,
               uint8_t* R, DevStatus* status) {
  const int jm = blockIdx.z % kOzModuli, split = blockIdx.z / kOzModuli;
  const int kbeg = split * kbs;
  const int nkb = max(0, min(kbs, nkb_total - kbeg));
  int m0, n0;
  pair_tile_coords(blockIdx.x, ntile, BN, &m0, &n0);
  ozm_pair_tile<false>(&mapA, &mapV, M, N, BN, col0, m0, n0, jm, kbeg, nkb,
                       R + (size_t)blockIdx.z * N * M, status);
}

// Grouped products: the tiles of up to kOzGroupMax independent problems in one launch
// (grid x runs over every problem's CTA pairs, z over the moduli); each problem has its own
// operands (tensor maps), sizes and residue buffer.  Used to batch the filter steps of many
// problems.
struct OzmGroupParams {
  CUtensorMap mapA[kOzGroupMax];
  CUtensorMap mapV[kOzGroupMax];
  void* R[kOzGroupMax];        // residues: one byte, or two (ring products)
  int ring[kOzGroupMax];       // 0: the real moduli; else the number of ring moduli
  int tile0[kOzGroupMax + 1];  // first grid-x CTA of each problem (even: pairs never straddle)
  int M[kOzGroupMax], N[kOzGroupMax], BN[kOzGroupMax], col0[kOzGroupMax], ntile[kOzGroupMax],
      nkb[kOzGroupMax];
  int count;
};
static_assert(sizeof(OzmGroupParams) <= 32000, "kernel parameter space");

__global__ void __launch_bounds__(M_THREADS, 1)
    ozm_group_kernel(const __grid_constant__ OzmGroupParams P, DevStatus* status) {
  int p = 0;
  while (p + 1 < P.count && (int)blockIdx.x >= P.tile0[p + 1]) ++p;
  const int jm = blockIdx.z;
  if (jm >= (P.ring[p] ? P.ring[p] : kOzModuli)) return;  // (the pair leaves together)
  int m0, n0;
  pair_tile_coords((int)blockIdx.x - P.tile0[p], P.ntile[p], P.BN[p], &m0, &n0);
  const size_t slab = (size_t)jm * P.N[p] * P.M[p];
  if (P.ring[p])
    ozm_pair_tile<true>(&P.mapA[p], &P.mapV[p], P.M[p], P.N[p], P.BN[p], P.col0[p], m0, n0, jm, 0,
                        P.nkb[p], (uint16_t*)P.R[p] + slab, status);
  else
    ozm_pair_tile<false>(&P.mapA[p], &P.mapV[p], P.M[p], P.N[p], P.BN[p], P.col0[p], m0, n0, jm, 0,
                         P.nkb[p], (uint8_t*)P.R[p] + slab, status);
}

// ---------------------------------------------------------------------------
// CRT reconstruction and epilogue:
//   v = 2^{e_r + f_c - 114} X,  X = CRT(residues) in (-P/2, P/2],
//   out64[r + (col0 + c) ldo] = alpha v + beta X64[.] + gamma Z64[.]  (same index).
// R holds `splits` partial residues per modulus; they are summed first.
// Integer-issue-bound: ~350 integer instructions per value.  All of the rounding and scaling is
// done on integers (an FP64 instruction takes 64 clocks of a sub-partition), only the update
// itself is FP64; a block takes rows of one column, so that no entry needs a division by M.
// n = 10000, 600 columns complex: 295 -> 175 us, real 171 -> 97 us.
// ---------------------------------------------------------------------------

// 2^e X rounded once to FP64, X = (sum_j r_j C_j, in 32-bit limbs with 64-bit headroom) mod P.
// |X| <= 0.39 P (the range checks beside the moduli: 2 K 2^114 against P / 2 and K <= 2^15 for 15
// ring moduli), and the FP32 quotient of the limbs' sum (< 2^15) by P is within 0.01, so the
// nearest integer to it is the right multiple of P.
template <class Tab>
__device__ __forceinline__ double crt_finish(const unsigned long long* acc, const Tab& tab, int e) {
  uint32_t x[5];
  unsigned long long carry = 0;
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    const unsigned long long t = acc[l] + carry;
    x[l] = (uint32_t)t;
    carry = t >> 32;
  }
  const float xf = (float)x[4] * 4294967296.0f + (float)x[3];  // X / 2^96, rounded
  const uint32_t q = (uint32_t)__float2int_rn(xf * tab.p96_over_P);
  uint32_t m[5];
  carry = 0;
#pragma unroll
  for (int l = 0; l < 5; ++l) {
    const unsigned long long t = (unsigned long long)tab.P[l] * q + carry;
    m[l] = (uint32_t)t;
    carry = t >> 32;
  }
  asm("sub.cc.u32 %0, %0, %5;\n\tsubc.cc.u32 %1, %1, %6;\n\tsubc.cc.u32 %2, %2, %7;\n\t"
      "subc.cc.u32 %3, %3, %8;\n\tsubc.u32 %4, %4, %9;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4])
      : "r"(m[0]), "r"(m[1]), "r"(m[2]), "r"(m[3]), "r"(m[4]));
  // magnitude and sign (two's complement, 160 bits)
  const uint32_t neg = (uint32_t)((int)x[4] >> 31);
#pragma unroll
  for (int l = 0; l < 5; ++l) x[l] ^= neg;
  asm("add.cc.u32 %0, %0, %5;\n\taddc.cc.u32 %1, %1, 0;\n\taddc.cc.u32 %2, %2, 0;\n\t"
      "addc.cc.u32 %3, %3, 0;\n\taddc.u32 %4, %4, 0;"
      : "+r"(x[0]), "+r"(x[1]), "+r"(x[2]), "+r"(x[3]), "+r"(x[4])
      : "r"(neg & 1u));
  // the leading word first: w0 w1 w2 and whether anything lies below
  uint32_t w0 = x[4], w1 = x[3], w2 = x[2], lo = x[1] | x[0];
  int base = 3;  // |X| = (w0 w1) 2^{32 base} + ...
  if (w0 == 0) { w0 = x[3]; w1 = x[2]; w2 = x[1]; lo = x[0]; base = 2; }
  if (w0 == 0) { w0 = x[2]; w1 = x[1]; w2 = x[0]; lo = 0; base = 1; }
  if (w0 == 0) { w0 = x[1]; w1 = x[0]; w2 = 0; base = 0; }
  if (w0 == 0) { w0 = x[0]; w1 = 0; base = -1; }
  if (w0 == 0) return 0.0;
  // 64 leading bits, normalised, with a sticky bit; rounded to 53, half to even
  const int lz = __clz((int)w0);
  const uint32_t h1 = __funnelshift_l(w1, w0, lz), h0 = __funnelshift_l(w2, w1, lz);
  const uint32_t sticky = ((w2 << lz) | lo) != 0 ? 1u : 0u;
  const unsigned long long hi = ((unsigned long long)h1 << 32) | h0 | sticky;
  const int sh = 32 * base - lz + e;  // |X| 2^e = hi 2^sh
  const int field = sh + 63 + 1023;   // exponent field of the result (before a carry)
  if (field < 1 || field > 2045) {
    const double v = ldexp(__ull2double_rn(hi), sh);
    return neg ? -v : v;
  }
  unsigned long long r = hi >> 11;
  const uint32_t low = (uint32_t)hi & 0x7FFu;
  r += (low > 0x400u || (low == 0x400u && (r & 1))) ? 1 : 0;
  // (the leading bit of r adds the 1 that the field is lowered by; a carry raises it)
  const unsigned long long bits = r + ((unsigned long long)(field - 1) << 52) + ((unsigned long long)(neg & 1u) << 63);
  return __longlong_as_double((long long)bits);
}

// The reconstruction of one product.
struct CrtItem {
  const void* R;
  const int *rowexp, *colexp;
  const double *X64, *Z64;
  double* out64;
  z64* zout;     // ring: complex output instead of the stacked one (zsub: subtracted from it)
  double alpha, beta, gamma;
  int M, N, col0, ldo, ring, zsub, splits;
  int blk0;      // first block of the item in a grouped launch
};

__device__ __forceinline__ void crt_update(const CrtItem& I, double v0, size_t idx) {
  double v = I.alpha * v0;
  if (I.beta != 0.0) v = fma(I.beta, I.X64[idx], v);
  if (I.gamma != 0.0) v = fma(I.gamma, I.Z64[idx], v);
  I.out64[idx] = v;
}

// E entries per thread: rows r .. r + E - 1 of column c (E > 1: M is a multiple of E).
constexpr int CRT_NT = 256;
__host__ __device__ inline int crt_blocks(int M, int N, int E) { return ((M + CRT_NT * E - 1) / (CRT_NT * E)) * N; }

// Real: residues of one byte.
template <int E>
__device__ __forceinline__ void crt_real(const CrtItem& I, int blk) {
  const int per = (I.M + CRT_NT * E - 1) / (CRT_NT * E), c = blk / per;
  const int r = ((blk - c * per) * CRT_NT + (int)threadIdx.x) * E;
  if (r >= I.M) return;
  const size_t plane = (size_t)I.M * I.N;
  const uint8_t* R = (const uint8_t*)I.R + (size_t)c * I.M + r;
  uint32_t w[kOzModuli], w2[kOzModuli];
#pragma unroll
  for (int j = 0; j < kOzModuli; ++j) {
    if constexpr (E == 4) {
      w[j] = *(const uint32_t*)(R + (size_t)j * plane);
      w2[j] = I.splits > 1 ? *(const uint32_t*)(R + (size_t)(kOzModuli + j) * plane) : 0u;
    } else {
      w[j] = R[(size_t)j * plane];
      w2[j] = I.splits > 1 ? R[(size_t)(kOzModuli + j) * plane] : 0u;
    }
  }
  const int ec = I.colexp[I.col0 + c] - 2 * OZ_KBITS;
#pragma unroll 1
  for (int k = 0; k < E; ++k) {
    unsigned long long acc[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < kOzModuli; ++j) {
      const uint32_t s = ((w[j] >> (8 * k)) & 0xFFu) + ((w2[j] >> (8 * k)) & 0xFFu);
#pragma unroll
      for (int l = 0; l < 5; ++l) acc[l] += (unsigned long long)s * c_crt.C[j][l];
    }
    crt_update(I, crt_finish(acc, c_crt, I.rowexp[r + k] + ec), (size_t)(r + k) + (size_t)(I.col0 + c) * I.ldo);
  }
}

// Ring: residues U | W of two bytes.
template <int NM, int E>
__device__ __forceinline__ void crt_ring(const CrtItem& I, int blk) {
  const int per = (I.M + CRT_NT * E - 1) / (CRT_NT * E), c = blk / per;
  const int r = ((blk - c * per) * CRT_NT + (int)threadIdx.x) * E;
  if (r >= I.M) return;
  const RingTable<NM>& tab = ring_table<NM>();
  const size_t plane = (size_t)I.M * I.N;
  const uint16_t* R = (const uint16_t*)I.R + (size_t)c * I.M + r;
  uint32_t u[NM], w[NM];
#pragma unroll
  for (int j = 0; j < NM; ++j) {
    if constexpr (E == 2) {
      u[j] = *(const uint32_t*)(R + (size_t)j * plane);
      w[j] = *(const uint32_t*)(R + (size_t)(NM + j) * plane);
    } else {
      u[j] = R[(size_t)j * plane];
      w[j] = R[(size_t)(NM + j) * plane];
    }
  }
  const int ec = I.colexp[I.col0 + c] - 2 * OZ_KBITS;
#pragma unroll 1
  for (int k = 0; k < E; ++k) {
    unsigned long long are[5] = {0, 0, 0, 0, 0}, aim[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < NM; ++j) {
      const uint32_t uj = (u[j] >> (16 * k)) & 0xFFFFu, wj = (w[j] >> (16 * k)) & 0xFFFFu;
      const uint32_t s = uj + wj, d = uj + (uint32_t)ring_modulus(j) - wj;
#pragma unroll
      for (int l = 0; l < 5; ++l) {
        are[l] += (unsigned long long)s * tab.Cre[j][l];
        aim[l] += (unsigned long long)d * tab.Cim[j][l];
      }
    }
    const int e = I.rowexp[r + k] + ec;
    const double re = crt_finish(are, tab, e), im = crt_finish(aim, tab, e);
    const size_t idx = (size_t)(r + k) + (size_t)(I.col0 + c) * I.ldo;
    if (I.zout) {
      z64 v{re, im};
      if (I.zsub) v = z64{I.zout[idx].x - re, I.zout[idx].y - im};
      I.zout[idx] = v;
    } else {
      crt_update(I, re, idx);
      crt_update(I, im, idx + I.M);
    }
  }
}

// KIND 1, 4: real, entries per thread; 15, 16: ring moduli, one entry; 30: 15 moduli, two entries.
template <int KIND>
__global__ void __launch_bounds__(CRT_NT) crt_kernel(const __grid_constant__ CrtItem I) {
  dep_wait();
  const int blk = blockIdx.x;
  if constexpr (KIND == 1 || KIND == 4) crt_real<KIND>(I, blk);
  else if constexpr (KIND == 30) crt_ring<kRingShort, 2>(I, blk);
  else crt_ring<KIND, 1>(I, blk);
}

struct CrtGroupParams {
  CrtItem it[kOzGroupMax];
  int count;
};
static_assert(sizeof(CrtGroupParams) <= 32000, "kernel parameter space");

__global__ void __launch_bounds__(CRT_NT) crt_group_kernel(const __grid_constant__ CrtGroupParams P) {
  dep_wait();
  int p = 0;
  while (p + 1 < P.count && (int)blockIdx.x >= P.it[p + 1].blk0) ++p;
  const CrtItem& I = P.it[p];
  const int blk = (int)blockIdx.x - I.blk0;
  if (I.ring == kRingShort) crt_ring<kRingShort, 1>(I, blk);
  else if (I.ring) crt_ring<kRingModuli, 1>(I, blk);
  else crt_real<1>(I, blk);
}

// Host: one product's reconstruction.  More entries per thread (wider loads) once every SM still
// has 2048 threads of them.
int crt_launch(cudaStream_t st, const CrtItem& I, int* launches) {
  const bool big = (long long)I.M * I.N >= 4LL * kNumSMs * 2048;
  if (I.ring == kRingShort) {
    if (big && I.M % 2 == 0) launch_dep(st, crt_blocks(I.M, I.N, 2), CRT_NT, 0, crt_kernel<30>, I);
    else launch_dep(st, crt_blocks(I.M, I.N, 1), CRT_NT, 0, crt_kernel<kRingShort>, I);
  } else if (I.ring) {
    launch_dep(st, crt_blocks(I.M, I.N, 1), CRT_NT, 0, crt_kernel<kRingModuli>, I);
  } else if (big && I.M % 4 == 0) {
    launch_dep(st, crt_blocks(I.M, I.N, 4), CRT_NT, 0, crt_kernel<4>, I);
  } else {
    launch_dep(st, crt_blocks(I.M, I.N, 1), CRT_NT, 0, crt_kernel<1>, I);
  }
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

// ---------------- residues of the integer operands ----------------

// |x| as its IEEE bit pattern: for non-negative doubles the integer order is the numeric
// order, so row / column maxima need no FP64 instructions (FP64 issues at 2 per clock per
// SM here, integer work at 64).
__device__ __forceinline__ unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

__device__ __forceinline__ int exp_bound(unsigned long long amax_bits) {
  // smallest e with amax < 2^e (0 for an all-zero row/column)
  if (amax_bits == 0) return 0;
  int e;
  frexp(__longlong_as_double((long long)amax_bits), &e);  // amax = f 2^e, f in [0.5, 1)
  return e;
}

// x_int = round(x 2^{57 - e}) (|x| < 2^e, so |x_int| <= 2^57), from the significand and
// exponent fields (round half away from zero: the integer of -x is minus that of x).
__device__ __forceinline__ long long oz_int(double x, int e) {
  const long long bits = __double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7FF);
  long long m = bits & ((1LL << 52) - 1);
  long long X = 0;
  if (ex != 0x7FF) {
    int sh;
    if (ex == 0) {
      sh = 1 - 1075 + OZ_KBITS - e;  // subnormal: x = m 2^-1074
    } else {
      m |= 1LL << 52;
      sh = ex - 1075 + OZ_KBITS - e;  // x = m 2^{ex - 1075}; |x| < 2^e gives m 2^sh < 2^57
    }
    if (sh >= 0) X = m << sh;
    else if (sh > -64) X = (m + (1LL << (-sh - 1))) >> (-sh);
    if (bits < 0) X = -X;
  }
  return X;
}

// Residues of four adjacent K entries (|X| < 2^58) mod p_j in [-(p/2), p - 1 - p/2], stored as BF16
// (exact: magnitudes <= 128), 8-byte words.  Cut up as in write_ring4 (below): one unreduced
// 31-bit sum and one division by a constant per residue (before: three divisions per residue and
// 2-byte stores).  Integer-issue-bound.  n = 4999, A 430 -> 235 us; a filter of 299 columns 9.95 ->
// 8.95 ms together with the split of columns below.
__device__ __forceinline__ void write_real4(const long long* x, __nv_bfloat16* base, size_t idx, size_t plane) {
  uint32_t x0[4], x1[4], x2[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const unsigned long long X = (unsigned long long)(x[d] + (1LL << 58));
    x0[d] = (uint32_t)X & 0x7FFFFu;
    x1[d] = (uint32_t)(X >> 19) & 0x7FFFFu;
    x2[d] = (uint32_t)(X >> 38);
  }
#pragma unroll
  for (int j = 0; j < kOzModuli; ++j) {
    const uint32_t p = (uint32_t)oz_modulus(j);
    const uint32_t k19 = (uint32_t)((1ull << 19) % p), k38 = (uint32_t)((1ull << 38) % p), half = p / 2;
    const uint32_t off = p - (uint32_t)((1ull << 58) % p) + half;
    float f[4];
#pragma unroll
    for (int d = 0; d < 4; ++d)  // < 2^21 2^8 + 2^19 2^8 + 2^19 + 2^9 < 2^30
      f[d] = (float)((int)((x2[d] * k38 + x1[d] * k19 + x0[d] + off) % p) - (int)half);
    __nv_bfloat162 pk[2] = {__floats2bfloat162_rn(f[0], f[1]), __floats2bfloat162_rn(f[2], f[3])};
    *(uint2*)(base + idx + (size_t)j * plane) = *(const uint2*)pk;
  }
}

// Ring residues of four adjacent K entries: u = (xr + s xi) mod p and w = (xr - s xi) mod p in
// symmetric range (|r| <= 254, exact in BF16), planes u then w, stored as 8-byte words.
// X + 2^58 >= 0 is cut into 21 | 19 | 19 bits, so X mod p needs one unreduced 31-bit sum of
// three products by constants and one division by a constant (the shift's class is taken off
// in the same sum): integer work bounds the slicing, not HBM.
template <int NM>
__device__ __forceinline__ void write_ring4(const long long* xr, const long long* xi, __nv_bfloat16* base,
                                            size_t idx, size_t plane) {
  uint32_t r0[4], r1[4], r2[4], i0[4], i1[4], i2[4];
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    const unsigned long long R = (unsigned long long)(xr[d] + (1LL << 58));
    const unsigned long long I = (unsigned long long)(xi[d] + (1LL << 58));
    r0[d] = (uint32_t)R & 0x7FFFFu;
    r1[d] = (uint32_t)(R >> 19) & 0x7FFFFu;
    r2[d] = (uint32_t)(R >> 38);
    i0[d] = (uint32_t)I & 0x7FFFFu;
    i1[d] = (uint32_t)(I >> 19) & 0x7FFFFu;
    i2[d] = (uint32_t)(I >> 38);
  }
#pragma unroll
  for (int j = 0; j < NM; ++j) {
    const uint32_t p = (uint32_t)ring_modulus(j), s = ring_root(j);
    const uint32_t k19 = (uint32_t)((1ull << 19) % p), k38 = (uint32_t)((1ull << 38) % p);
    const uint32_t off = p - (uint32_t)((1ull << 58) % p), half = p / 2;
    float fu[4], fw[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      // < 2^21 2^9 + 2^19 2^9 + 2^19 + 2^9 < 2^31, and + s ti < 2^18
      const uint32_t tr = r2[d] * k38 + r1[d] * k19 + r0[d] + off;
      const uint32_t ti = (i2[d] * k38 + i1[d] * k19 + i0[d] + off) % p;
      const uint32_t u = tr + s * ti + half, w = tr + (p - s) * ti + half;
      fu[d] = (float)((int)(u % p) - (int)half);
      fw[d] = (float)((int)(w % p) - (int)half);
    }
    const size_t at = idx + (size_t)j * plane;
    __nv_bfloat162 pk[2];
    pk[0] = __floats2bfloat162_rn(fu[0], fu[1]);
    pk[1] = __floats2bfloat162_rn(fu[2], fu[3]);
    *(uint2*)(base + at) = *(const uint2*)pk;
    pk[0] = __floats2bfloat162_rn(fw[0], fw[1]);
    pk[1] = __floats2bfloat162_rn(fw[2], fw[3]);
    *(uint2*)(base + (size_t)NM * plane + at) = *(const uint2*)pk;
  }
}

__device__ __forceinline__ unsigned long long block_max(unsigned long long v, unsigned long long* red) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
  __syncthreads();
  if (lane == 0) red[wi] = v;
  __syncthreads();
  unsigned long long mx = 0;
  for (int i = 0; i < nw; ++i) mx = red[i] > mx ? red[i] : mx;
  return mx;
}

// Exponent of n values, by the whole block.
__device__ __forceinline__ int column_exp(const double* col, int n, unsigned long long* red) {
  unsigned long long amax = 0;
#pragma unroll 4
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const unsigned long long b = abs_bits(col[k]);
    amax = b > amax ? b : amax;
  }
  return exp_bound(block_max(amax, red));
}

// Residues of entries [k0, k1) of a column of n values (multiples of 4; zero from n on), at idx + k.
__device__ __forceinline__ void slice_real(const double* col, int n, int k0, int k1, int e,
                                           __nv_bfloat16* planes, size_t idx, size_t plane) {
  for (int k = k0 + 4 * threadIdx.x; k < k1; k += 4 * blockDim.x) {
    long long x[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) x[d] = oz_int(k + d < n ? col[k + d] : 0.0, e);
    write_real4(x, planes, idx + k, plane);
  }
}

// A column is sliced by `parts` blocks, each of which takes its exponent for itself (an L2 read of
// the column): one block per column leaves most of the SMs' warps empty for few columns, and half of
// them at 600.  A part is at least 1024 rows, four per thread.
__host__ __device__ inline int slice_part(int kp, int parts) { return (kp / 64 + parts - 1) / parts * 64; }
inline int slice_parts(int kp, int cols) {
  return std::max(1, std::min(kp / 1024, 8 * kNumSMs / std::max(1, cols)));
}

// Real A (n x n): residues of row m (column m of A: symmetric) into planes (row-major, ld kp),
// row exponent into rowexp[m].
__global__ void __launch_bounds__(256) oz_slice_A_kernel(int n, const double* A, int lda,
                                                         int kp, __nv_bfloat16* planes,
                                                         size_t plane, int* rowexp) {
  dep_wait();
  __shared__ unsigned long long red[8];
  const int m = blockIdx.x;
  const double* col = A + (size_t)m * lda;
  const int e = column_exp(col, n, red);
  if (threadIdx.x == 0) rowexp[m] = e;
  slice_real(col, n, 0, kp, e, planes, (size_t)m * kp, plane);
}

// FP64 stacked block V64 (M x ncols, ld ldi): residues of column c into planes
// (column-major, ld kp; rows >= M zero), column exponent into colexp[c].
__global__ void __launch_bounds__(256) oz_slice_V_kernel(int M, int c0, const double* V64,
                                                         int ldi, int kp, __nv_bfloat16* planes,
                                                         size_t plane, int* colexp) {
  dep_wait();
  __shared__ unsigned long long red[8];
  const int c = c0 + blockIdx.x, part = slice_part(kp, gridDim.y), k0 = blockIdx.y * part;
  const double* col = V64 + (size_t)c * ldi;
  const int e = column_exp(col, M, red);
  if (threadIdx.x == 0 && blockIdx.y == 0) colexp[c] = e;
  slice_real(col, M, k0, min(kp, k0 + part), e, planes, (size_t)c * kp, plane);
}

// ---- operands of the ring products ----
// The row exponents of A (over Re and Im together) and the column exponents of V are those of
// the stacked form, and so are the integers of Ar, Ai, Vr, Vi.  Layout: two plane sets (u | w),
// each NM planes of one row per row of A (column of V), K contiguous.

// Row m of A (complex Hermitian, column-major): its integer row from column m of A
// (A[m, k] = conj(A[k, m])): Ar[m, k] = Re A[k, m], Ai[m, k] = -Im A[k, m].
template <int NM>
__global__ void __launch_bounds__(256) oz_slice_A_ring_kernel(int n, const z64* A, int lda,
                                                              int kpn, __nv_bfloat16* planes, size_t plane,
                                                              int* rowexp) {
  dep_wait();
  __shared__ unsigned long long red[8];
  const int m = blockIdx.x;
  const z64* col = A + (size_t)m * lda;
  unsigned long long amax = 0;
  for (int k = threadIdx.x; k < n; k += 256) {
    const unsigned long long b = max(abs_bits(col[k].x), abs_bits(col[k].y));
    amax = b > amax ? b : amax;
  }
  const int e = exp_bound(block_max(amax, red));
  if (threadIdx.x == 0) rowexp[m] = e;
  for (int k = 4 * threadIdx.x; k < kpn; k += 1024) {  // kpn is a multiple of 64
    long long xr[4], xi[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const z64 a = (k + d < n) ? col[k + d] : z64{0.0, 0.0};
      xr[d] = oz_int(a.x, e);
      xi[d] = -oz_int(a.y, e);
    }
    write_ring4<NM>(xr, xi, planes, (size_t)m * kpn + k, plane);
  }
}

// Column c of the stacked FP64 block V64 ([Re V; Im V], 2n rows, ld ldi): its exponent over
// both halves, then its two plane rows (u | w), ld kpn.
template <int NM>
__device__ __forceinline__ void slice_V_ring_column(int n, int c, const double* V64, int ldi,
                                                    int kpn, int k0, int k1, __nv_bfloat16* planes,
                                                    size_t plane, int* colexp, unsigned long long* red) {
  const double* col = V64 + (size_t)c * ldi;
  const int e = column_exp(col, 2 * n, red);
  if (threadIdx.x == 0 && k0 == 0) colexp[c] = e;
  for (int k = k0 + 4 * threadIdx.x; k < k1; k += 1024) {
    long long xr[4], xi[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const bool in = k + d < n;
      xr[d] = oz_int(in ? col[k + d] : 0.0, e);
      xi[d] = oz_int(in ? col[n + k + d] : 0.0, e);
    }
    write_ring4<NM>(xr, xi, planes, (size_t)c * kpn + k, plane);
  }
}

// Grouped form of oz_slice_V_kernel: parts[p] blocks per sliced column of every problem.
struct SliceGroupParams {
  const double* V64[kOzGroupMax];
  __nv_bfloat16* planes[kOzGroupMax];
  int* colexp[kOzGroupMax];
  long long plane[kOzGroupMax];
  int blk0[kOzGroupMax + 1];  // first block of each problem
  int M[kOzGroupMax], c0[kOzGroupMax], ldi[kOzGroupMax], kp[kOzGroupMax];
  int ring[kOzGroupMax];  // ring moduli of a complex problem (M = n); 0: real
  int parts[kOzGroupMax];
  int count;
};
static_assert(sizeof(SliceGroupParams) <= 32000, "kernel parameter space");

__global__ void __launch_bounds__(256) oz_slice_V_group_kernel(const __grid_constant__ SliceGroupParams P) {
  dep_wait();
  __shared__ unsigned long long red[8];
  int p = 0;
  while (p + 1 < P.count && (int)blockIdx.x >= P.blk0[p + 1]) ++p;
  const int b = blockIdx.x - P.blk0[p], c = P.c0[p] + b / P.parts[p];
  const int M = P.M[p], kp = P.kp[p];
  const int part = slice_part(kp, P.parts[p]), k0 = b % P.parts[p] * part, k1 = min(kp, k0 + part);
  if (P.ring[p]) {
    if (P.ring[p] == kRingShort)
      slice_V_ring_column<kRingShort>(M, c, P.V64[p], P.ldi[p], kp, k0, k1, P.planes[p], (size_t)P.plane[p],
                                      P.colexp[p], red);
    else
      slice_V_ring_column<kRingModuli>(M, c, P.V64[p], P.ldi[p], kp, k0, k1, P.planes[p], (size_t)P.plane[p],
                                       P.colexp[p], red);
    return;
  }
  const double* col = P.V64[p] + (size_t)c * P.ldi[p];
  const int e = column_exp(col, M, red);
  if (threadIdx.x == 0 && k0 == 0) P.colexp[p][c] = e;
  slice_real(col, M, k0, k1, e, P.planes[p], (size_t)c * kp, (size_t)P.plane[p]);
}

// Caller's block V (n x ncols, ld ldv) -> stacked FP64 (M x ncols, ld ldo).
template <class T>
__global__ void stack_V_kernel(int n, int ncols, const T* V, int ldv, double* V64,
                               int ldo) {
  dep_wait();
  const int M = Sc<T>::cplx ? 2 * n : n;
  const size_t total = (size_t)M * ncols;
  for (size_t t = blockIdx.x * (size_t)blockDim.x + threadIdx.x; t < total;
       t += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % M), a = (int)(t / M);
    double x;
    if constexpr (Sc<T>::cplx) {
      const z64 v = V[(size_t)(i % n) + (size_t)a * ldv];
      x = (i < n) ? v.x : v.y;
    } else {
      x = V[(size_t)i + (size_t)a * ldv];
    }
    V64[(size_t)i + (size_t)a * ldo] = x;
  }
}

// Column blockIdx.x of a complex block Y (n x q, ld ldy): its exponent (over Re and Im) and its
// two plane rows (u | w), ld kp; entries past n are zero.
template <int NM>
__global__ void __launch_bounds__(256) oz_slice_cols_ring_kernel(int n, const z64* Y, int ldy, int kp,
                                                                 __nv_bfloat16* planes, size_t plane,
                                                                 int* colexp) {
  dep_wait();
  __shared__ unsigned long long red[8];
  const int c = blockIdx.x, part = slice_part(kp, gridDim.y), k0 = blockIdx.y * part, k1 = min(kp, k0 + part);
  const z64* col = Y + (size_t)c * ldy;
  unsigned long long amax = 0;
#pragma unroll 4
  for (int k = threadIdx.x; k < n; k += 256) {
    const unsigned long long b = max(abs_bits(col[k].x), abs_bits(col[k].y));
    amax = b > amax ? b : amax;
  }
  const int e = exp_bound(block_max(amax, red));
  if (threadIdx.x == 0 && k0 == 0) colexp[c] = e;
  for (int k = k0 + 4 * threadIdx.x; k < k1; k += 1024) {
    long long xr[4], xi[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const z64 a = (k + d < n) ? col[k + d] : z64{0.0, 0.0};
      xr[d] = oz_int(a.x, e);
      xi[d] = oz_int(a.y, e);
    }
    write_ring4<NM>(xr, xi, planes, (size_t)c * kp + k, plane);
  }
}

// Row exponents (over Re and Im) of a column-major complex X (n x l): 32 rows per CTA, eight
// column groups.
__global__ void __launch_bounds__(256) oz_row_exp_kernel(int n, int l, const z64* X, int ldx,
                                                         int* rowexp) {
  dep_wait();
  __shared__ unsigned long long red[8][32];
  const int i = threadIdx.x & 31, g = threadIdx.x >> 5, r = blockIdx.x * 32 + i;
  unsigned long long m = 0;
  if (r < n)
    for (int k = g; k < l; k += 8) {
      const z64 a = X[(size_t)r + (size_t)k * ldx];
      const unsigned long long b = max(abs_bits(a.x), abs_bits(a.y));
      m = b > m ? b : m;
    }
  red[g][i] = m;
  __syncthreads();
  if (g == 0 && r < n) {
    for (int j = 1; j < 8; ++j) m = red[j][i] > m ? red[j][i] : m;
    rowexp[r] = exp_bound(m);
  }
}

// Rows of a column-major complex X (n x l) as plane rows (u | w, ld kp, K contiguous): 32 rows
// x 64 of K per CTA through shared memory, so that X is read along its columns and the planes
// are written along K.
template <int NM>
__global__ void __launch_bounds__(256) oz_slice_rows_ring_kernel(int n, int l, const z64* X, int ldx,
                                                                 int kp, __nv_bfloat16* planes, size_t plane,
                                                                 const int* rowexp) {
  dep_wait();
  __shared__ z64 tile[64][33];
  const int r0 = blockIdx.x * 32, k0 = blockIdx.y * 64;
  const int i = threadIdx.x & 31, g = threadIdx.x >> 5;
  for (int k = g; k < 64; k += 8)
    tile[k][i] = (r0 + i < n && k0 + k < l) ? X[(size_t)(r0 + i) + (size_t)(k0 + k) * ldx] : z64{0.0, 0.0};
  __syncthreads();
  for (int t = threadIdx.x; t < 512; t += 256) {
    const int row = t >> 4, k = 4 * (t & 15);
    if (r0 + row >= n) continue;
    const int e = rowexp[r0 + row];
    long long xr[4], xi[4];
#pragma unroll
    for (int d = 0; d < 4; ++d) {
      const z64 a = tile[k + d][row];
      xr[d] = oz_int(a.x, e);
      xi[d] = oz_int(a.y, e);
    }
    write_ring4<NM>(xr, xi, planes, (size_t)(r0 + row) * kp + k0 + k, plane);
  }
}

// Xt (l x n, ld ldt) is the transpose of a real column-major X (n x l): row m of X is column m
// of Xt.  Residues of the rows into planes (row-major, ld kp), row exponents into rowexp.
__global__ void __launch_bounds__(256) oz_slice_rows_kernel(int l, const double* Xt, int ldt, int kp,
                                                            __nv_bfloat16* planes, size_t plane, int* rowexp) {
  dep_wait();
  __shared__ unsigned long long red[8];
  const int m = blockIdx.x;
  const double* row = Xt + (size_t)m * ldt;  // X[m, 0..l)
  const int e = column_exp(row, l, red);
  if (threadIdx.x == 0) rowexp[m] = e;
  slice_real(row, l, 0, kp, e, planes, (size_t)m * kp, plane);
}

// Residues of the columns of a real block Y (n x q, ld ldy): planes column-major (ld kp; rows
// >= n are zero), column exponents.
__global__ void __launch_bounds__(256) oz_slice_cols_kernel(int n, const double* Y, int ldy, int kp,
                                                            __nv_bfloat16* planes, size_t plane, int* colexp) {
  dep_wait();
  __shared__ unsigned long long red[8];
  const int j = blockIdx.x, part = slice_part(kp, gridDim.y), k0 = blockIdx.y * part;
  const double* col = Y + (size_t)j * ldy;
  const int e = column_exp(col, n, red);
  if (threadIdx.x == 0 && k0 == 0) colexp[j] = e;
  slice_real(col, n, k0, min(kp, k0 + part), e, planes, (size_t)j * kp, plane);
}

// Xt = X^T: real X n x l (ld ldx) -> Xt l x n (ld ldt).
__global__ void transpose_kernel(int n, int l, const double* X, int ldx, double* Xt, int ldt) {
  dep_wait();
  __shared__ double tile[32][33];
  const int i0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int i = i0 + threadIdx.x, j = j0 + r;
    if (i < n && j < l) tile[r][threadIdx.x] = X[(size_t)i + (size_t)j * ldx];
  }
  __syncthreads();
  for (int r = threadIdx.y; r < 32; r += blockDim.y) {
    const int j = j0 + threadIdx.x, i = i0 + r;
    if (i < n && j < l) Xt[(size_t)j + (size_t)i * ldt] = tile[threadIdx.x][r];
  }
}

PFN_cuTensorMapEncodeTiled_v12000 encoder() {
  // looked up once (thread-safe static initialisation: batch sessions call from several threads)
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return (PFN_cuTensorMapEncodeTiled_v12000)p;
    return nullptr;
  }();
  return fn;
}

// 3-D BF16 map over the residue planes: {kp (contiguous), rows, planes}, box {64, box_rows, 1},
// 128-byte swizzle; consecutive planes are plane_rows * kp elements apart.
int make_map3(CUtensorMap* map, const void* base, int kp, int rows, int plane_rows, int box_rows,
              int planes = kOzModuli) {
  auto enc = encoder();
  if (!enc) return CHASE_ERR_CUDA;
  cuuint64_t dims[3] = {(cuuint64_t)kp, (cuuint64_t)rows, (cuuint64_t)planes};
  cuuint64_t strides[2] = {(cuuint64_t)kp * 2, (cuuint64_t)kp * 2 * (cuuint64_t)plane_rows};
  cuuint32_t box[3] = {MBK, (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides,
                   box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : CHASE_ERR_CUDA;
}

}  // namespace

size_t ring_residue_bytes(int n, int kpn, int N) {
  return (size_t)2 * ring_moduli(kpn) * sizeof(uint16_t) * (size_t)n * (size_t)N;
}

size_t oz_residue_bytes(int M, int N) {
  return (size_t)kOzMaxSplits * kOzModuli * (size_t)M * (size_t)N;
}

int oz_slice_A(cudaStream_t st, int n, const double* A, int lda, int kp, void* planes, int* rowexp,
               int* launches) {
  launch_dep(st, n, 256, 0, oz_slice_A_kernel, n, A, lda, kp, (__nv_bfloat16*)planes, (size_t)n * kp, rowexp);
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

int oz_slice_A_ring(cudaStream_t st, int n, const z64* A, int lda, int kpn, void* planes, int* rowexp,
                    int* launches) {
  const size_t plane = (size_t)n * kpn;
  if (ring_moduli(kpn) == kRingShort)
    launch_dep(st, n, 256, 0, oz_slice_A_ring_kernel<kRingShort>, n, A, lda, kpn, (__nv_bfloat16*)planes, plane,
               rowexp);
  else
    launch_dep(st, n, 256, 0, oz_slice_A_ring_kernel<kRingModuli>, n, A, lda, kpn, (__nv_bfloat16*)planes, plane,
               rowexp);
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

int oz_slice_V(cudaStream_t st, int M, int c0, int c1, const double* V64, int ldi, int kp,
               int ncols_total, void* planes, int* colexp, int* launches) {
  if (c1 <= c0) return 0;
  launch_dep(st, dim3(c1 - c0, slice_parts(kp, c1 - c0)), 256, 0, oz_slice_V_kernel, M, c0, V64, ldi, kp, (__nv_bfloat16*)planes,
             (size_t)ncols_total * kp, colexp);
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

namespace {

// Launch with clusters of two CTAs along x (the CTA pairs of the modular products).
template <class... Params, class... Args>
int launch_pairs(void (*kernel)(Params...), dim3 grid, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(M_THREADS);
  cfg.dynamicSmemBytes = M_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_dep
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  CHASE_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, args...));
  return 0;
}

// The modular products of one plan; returns the number of K splits their residues hold in
// *splits.
int ozm_launch(cudaStream_t st, int M, int kp, const void* Aplanes, int a_plane_rows,
               const void* Vplanes, int ncols_total, int col0, int N, DevStatus* dst,
               Scratch resbuf, int* launches, const OzPlan& plan, int* splits) {
  if (a_plane_rows < M) a_plane_rows = M;
  // column tiles of at most plan.bn_max (a multiple of 16), as even as possible
  const int ntile = ceil_div(N, std::min(plan.bn_max, MBN_MAX));
  const int BN = ceil_div(ceil_div(N, ntile), 16) * 16;
  CUtensorMap mA, mV;
  if (make_map3(&mA, Aplanes, kp, M, a_plane_rows, MBM) ||
      make_map3(&mV, Vplanes, kp, ncols_total, ncols_total, tile_shape(BN).h0 / 2))
    return CHASE_ERR_CUDA;
  CHASE_CUDA_TRY(cudaFuncSetAttribute(ozm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, M_SMEM));
  const int nkb = kp / MBK;
  const int mblk = ceil_div(M, 2 * MBM) * 2;  // 128-row blocks, an even number (CTA pairs)
  const size_t slab = (size_t)kOzModuli * (size_t)M * N;  // residue bytes of one split
  // split K (whole 1024-wide chunks) until there are about four waves of CTAs
  constexpr int kChunkKB = 1024 / MBK;  // K blocks of one exact chunk
  const int nchunks = ceil_div(nkb, kChunkKB);
  int S = std::max(1, std::min(nchunks, ceil_div(4 * kNumSMs, ntile * mblk * kOzModuli)));
  if (plan.splits > 0) S = std::min(plan.splits, nchunks);
  // no split longer than kOzSplitMaxK (the range of the epilogue's exact reduction)
  const int min_S = ceil_div(nchunks, kOzSplitMaxK / 1024);
  S = std::max(std::min(S, kOzMaxSplits), min_S);
  while (S > min_S && (size_t)S * slab > resbuf.bytes) --S;
  if ((size_t)S * slab > resbuf.bytes) return CHASE_ERR_OOM;
  const int kbs = ceil_div(nchunks, S) * kChunkKB;  // whole chunks
  S = ceil_div(nkb, kbs);
  TRY_OZ(launch_pairs(ozm_kernel, dim3(ntile * mblk, 1, kOzModuli * S), st, mA, mV, M, N, BN, ntile,
                      col0, nkb, kbs, (uint8_t*)resbuf.ptr, dst));
  if (launches) ++*launches;
  *splits = S;
  return 0;
}

}  // namespace

int oz_gemm(cudaStream_t st, int M, int kp, const void* Aplanes, const int* rowexp,
            int a_plane_rows, const void* Vplanes, const int* colexp, int ncols_total, int col0,
            int N, double alpha, double beta, const double* X64, double gamma, const double* Z64,
            double* out64, int ldo, DevStatus* dst, Scratch resbuf, int* launches, int tune,
            int* trials) {
  if (N <= 0 || M <= 0) return 0;
  if (kp % MBK != 0 || kp > kOzMaxK) return CHASE_ERR_UNSUPPORTED;
  OzPlan plan;
  const bool known = oz_plan_lookup(M, N, kp, 0, &plan);
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (tune && !known && cudaStreamIsCapturing(st, &cs) == cudaSuccess &&
      cs == cudaStreamCaptureStatusNone) {
    // time the modular products of every candidate plan (they read only the residue planes
    // and all yield the same exact residues), keep the fastest, then run it once more and
    // reconstruct: the three-term update, which may read its own output, runs once
    OzPlan cand[6];
    const int nc = oz_plan_candidates(N, cand, 6);
    cudaEvent_t ev[7];
    for (int i = 0; i <= nc; ++i) CHASE_CUDA_TRY(cudaEventCreate(&ev[i]));
    int rc = 0, S = 1;
    cudaEventRecord(ev[0], st);
    for (int i = 0; i < nc && !rc; ++i) {
      rc = ozm_launch(st, M, kp, Aplanes, a_plane_rows, Vplanes, ncols_total, col0, N, dst, resbuf,
                      launches, cand[i], &S);
      cudaEventRecord(ev[i + 1], st);
    }
    if (!rc && cudaEventSynchronize(ev[nc]) == cudaSuccess) {
      int best = 0;
      float tbest = 1e30f;
      for (int i = 0; i < nc; ++i) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev[i], ev[i + 1]);
        if (ms < tbest) { tbest = ms; best = i; }
      }
      oz_plan_store(M, N, kp, 0, cand[best], tbest * 1e-3);
      if (trials) *trials += nc;
      plan = cand[best];
    }
    for (int i = 0; i <= nc; ++i) cudaEventDestroy(ev[i]);
    if (rc) return rc;
  }
  int S = 1;
  TRY_OZ(ozm_launch(st, M, kp, Aplanes, a_plane_rows, Vplanes, ncols_total, col0, N, dst, resbuf,
                    launches, plan, &S));
  CrtItem I{};
  I.R = resbuf.ptr;
  I.rowexp = rowexp;
  I.colexp = colexp;
  I.X64 = X64;
  I.Z64 = Z64;
  I.out64 = out64;
  I.alpha = alpha;
  I.beta = beta;
  I.gamma = gamma;
  I.M = M;
  I.N = N;
  I.col0 = col0;
  I.ldo = ldo;
  I.splits = S;
  return crt_launch(st, I, launches);
}

int oz_slice_V_group(cudaStream_t st, int count, const OzGroupItem* items, int* launches) {
  for (int g0 = 0; g0 < count; g0 += kOzGroupMax) {
    const int cnt = std::min(kOzGroupMax, count - g0);
    SliceGroupParams P{};
    int blocks = 0, cols = 0;
    for (int i = 0; i < cnt; ++i) cols += std::max(0, items[g0 + i].N);
    P.count = 0;
    for (int i = 0; i < cnt; ++i) {
      const OzGroupItem& it = items[g0 + i];
      if (it.N <= 0) continue;
      const int p = P.count++;
      P.V64[p] = it.V64_in;
      P.planes[p] = (__nv_bfloat16*)const_cast<void*>(it.Vplanes);
      P.colexp[p] = const_cast<int*>(it.colexp);
      P.plane[p] = (long long)it.ncols_total * it.kp;
      P.blk0[p] = blocks;
      P.parts[p] = slice_parts(it.kp, cols);
      P.M[p] = it.M;
      P.c0[p] = it.col0;
      P.ldi[p] = it.ldi;
      P.kp[p] = it.kp;
      P.ring[p] = it.ring ? ring_moduli(it.kp) : 0;
      blocks += it.N * P.parts[p];
    }
    if (P.count == 0) continue;
    P.blk0[P.count] = blocks;
    launch_dep(st, blocks, 256, 0, oz_slice_V_group_kernel, P);
    if (launches) ++*launches;
    CHASE_CUDA_TRY(cudaGetLastError());
  }
  return 0;
}

namespace {

// Appends the modular products of one item (its one or two plane sets) to a grouped launch.
int ozm_append(OzmGroupParams& P, int& tiles, const OzGroupItem& it, int bn_max) {
  const int sets = it.ring ? 2 : 1;  // ring products: U, W
  const int nm = it.ring ? ring_moduli(it.kp) : kOzModuli;
  const int ntile = ceil_div(it.N, std::min(bn_max, MBN_MAX));
  const int BN = ceil_div(ceil_div(it.N, ntile), 16) * 16;
  const int rows = std::max(it.a_plane_rows, it.M);
  const size_t rset = (size_t)nm * (it.ring ? 2 : 1) * it.M * it.N;  // residue bytes of one set
  const size_t aset = (size_t)nm * rows * it.kp * 2;                 // bytes of one A plane set
  const size_t vset = (size_t)nm * it.ncols_total * it.kp * 2;       // of one V plane set
  if (sets * rset > it.resbuf.bytes) return CHASE_ERR_OOM;
  for (int sidx = 0; sidx < sets; ++sidx) {
    const int p = P.count++;
    if (make_map3(&P.mapA[p], (const char*)it.Aplanes + (sidx ^ it.aswap) * aset, it.kp, it.M, rows, MBM, nm) ||
        make_map3(&P.mapV[p], (const char*)it.Vplanes + sidx * vset, it.kp, it.ncols_total,
                  it.ncols_total, tile_shape(BN).h0 / 2, nm))
      return CHASE_ERR_CUDA;
    P.R[p] = (char*)it.resbuf.ptr + sidx * rset;
    P.ring[p] = it.ring ? nm : 0;
    P.tile0[p] = tiles;
    P.M[p] = it.M;
    P.N[p] = it.N;
    P.BN[p] = BN;
    P.col0[p] = it.col0;
    P.ntile[p] = ntile;
    P.nkb[p] = it.kp / MBK;
    tiles += ntile * ceil_div(it.M, 2 * MBM) * 2;  // CTA pairs over 256-row blocks
  }
  return 0;
}

int ozm_launch_group(cudaStream_t st, OzmGroupParams& P, int tiles, DevStatus* dst, int* launches) {
  P.tile0[P.count] = tiles;
  int planes = 0;  // moduli of the longest set in the launch
  for (int p = 0; p < P.count; ++p) planes = std::max(planes, P.ring[p] ? P.ring[p] : kOzModuli);
  TRY_OZ(launch_pairs(ozm_group_kernel, dim3(tiles, 1, planes), st, P, dst));
  if (launches) ++*launches;
  return 0;
}

// Times one item's modular products with every candidate tile width (they read only the
// residue planes and all yield the same exact residues) and records the fastest.
int tune_group_item(cudaStream_t st, const OzGroupItem& it, DevStatus* dst, int* launches, int* trials) {
  OzPlan cand[6];
  const int all = oz_plan_candidates(it.N, cand, 6);
  int nc = 0;
  for (int i = 0; i < all; ++i)
    if (cand[i].splits == 1) cand[nc++] = cand[i];  // K is not split in a grouped launch
  cudaEvent_t ev[7];
  for (int i = 0; i <= nc; ++i) CHASE_CUDA_TRY(cudaEventCreate(&ev[i]));
  int rc = 0;
  cudaEventRecord(ev[0], st);
  for (int i = 0; i < nc && !rc; ++i) {
    OzmGroupParams P{};
    int tiles = 0;
    rc = ozm_append(P, tiles, it, cand[i].bn_max);
    if (!rc) rc = ozm_launch_group(st, P, tiles, dst, launches);
    cudaEventRecord(ev[i + 1], st);
  }
  if (!rc && cudaEventSynchronize(ev[nc]) == cudaSuccess) {
    int best = 0;
    float tbest = 1e30f;
    for (int i = 0; i < nc; ++i) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[i], ev[i + 1]);
      if (ms < tbest) { tbest = ms; best = i; }
    }
    oz_plan_store(it.M, it.N, it.kp, it.ring ? ring_moduli(it.kp) : 0, cand[best], tbest * 1e-3);
    if (trials) *trials += nc;
  }
  for (int i = 0; i <= nc; ++i) cudaEventDestroy(ev[i]);
  return rc;
}

}  // namespace

int oz_gemm_group(cudaStream_t st, int count, const OzGroupItem* items, DevStatus* dst, int* launches, int tune,
                  int* trials) {
  CHASE_CUDA_TRY(cudaFuncSetAttribute(ozm_group_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, M_SMEM));
  OzmGroupParams P{};
  CrtGroupParams C{};
  int tiles = 0;
  int blocks = 0;
  // one launch of the modular products and one of the reconstructions for what is gathered
  auto flush = [&]() -> int {
    if (P.count == 0) return 0;
    TRY_OZ(ozm_launch_group(st, P, tiles, dst, launches));
    if (C.count == 1) {
      TRY_OZ(crt_launch(st, C.it[0], launches));
    } else {
      launch_dep(st, blocks, CRT_NT, 0, crt_group_kernel, C);
      if (launches) ++*launches;
      CHASE_CUDA_TRY(cudaGetLastError());
    }
    P = OzmGroupParams{};
    C = CrtGroupParams{};
    tiles = 0;
    blocks = 0;
    return 0;
  };
  for (int i = 0; i < count; ++i) {
    const OzGroupItem& it = items[i];
    if (it.N <= 0 || it.M <= 0) continue;
    if (it.kp % MBK != 0 || it.kp > kOzSplitMaxK) return CHASE_ERR_UNSUPPORTED;  // K is not split here
    if (P.count + (it.ring ? 2 : 1) > kOzGroupMax || C.count + 1 > kOzGroupMax) TRY_OZ(flush());
    OzPlan plan;  // the autotuner's tile width for this shape, if it measured one
    const int kind = it.ring ? ring_moduli(it.kp) : 0;
    const bool known = oz_plan_lookup(it.M, it.N, it.kp, kind, &plan);
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (tune && !known && count == 1 && cudaStreamIsCapturing(st, &cs) == cudaSuccess &&
        cs == cudaStreamCaptureStatusNone) {
      TRY_OZ(tune_group_item(st, it, dst, launches, trials));
      oz_plan_lookup(it.M, it.N, it.kp, kind, &plan);
    }
    TRY_OZ(ozm_append(P, tiles, it, plan.bn_max));
    CrtItem& I = C.it[C.count++];
    I.R = it.resbuf.ptr;
    I.rowexp = it.rowexp;
    I.colexp = it.colexp;
    I.X64 = it.X64;
    I.Z64 = it.Z64;
    I.out64 = it.out64;
    I.zout = it.zout;
    I.alpha = it.alpha;
    I.beta = it.beta;
    I.gamma = it.gamma;
    I.M = it.M;
    I.N = it.N;
    I.col0 = it.col0;
    I.ldo = it.ldo;
    I.ring = it.ring ? ring_moduli(it.kp) : 0;
    I.zsub = it.zsub;
    I.splits = 1;
    I.blk0 = blocks;
    blocks += crt_blocks(it.M, it.N, 1);
  }
  return flush();
}

template <class T>
int oz_stack_V(cudaStream_t st, int n, int ncols, const T* V, int ldv, double* V64, int ldo,
               int* launches) {
  if (ncols <= 0) return 0;
  const int M = Sc<T>::cplx ? 2 * n : n;
  const size_t work = (size_t)M * ncols;
  const int blocks = (int)std::max<size_t>(1, std::min<size_t>((work + 255) / 256, (size_t)kNumSMs * 16));
  launch_dep(st, blocks, 256, 0, stack_V_kernel<T>, n, ncols, V, ldv, V64, ldo);
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

int oz_slice_cols_ring(cudaStream_t st, int n, int q, const z64* Y, int ldy, int kp, void* planes, int* colexp,
                       int* launches) {
  if (q <= 0) return 0;
  auto kern = ring_moduli(kp) == kRingShort ? oz_slice_cols_ring_kernel<kRingShort> : oz_slice_cols_ring_kernel<kRingModuli>;
  launch_dep(st, dim3(q, slice_parts(kp, q)), 256, 0, kern, n, Y, ldy, kp, (__nv_bfloat16*)planes, (size_t)q * kp, colexp);
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

int oz_slice_rows_ring(cudaStream_t st, int n, int l, const z64* X, int ldx, int kp, void* planes, int* rowexp,
                       int* launches) {
  if (n <= 0) return 0;
  launch_dep(st, ceil_div(n, 32), 256, 0, oz_row_exp_kernel, n, l, X, ldx, rowexp);
  auto kern = ring_moduli(kp) == kRingShort ? oz_slice_rows_ring_kernel<kRingShort> : oz_slice_rows_ring_kernel<kRingModuli>;
  launch_dep(st, dim3(ceil_div(n, 32), kp / 64), 256, 0, kern, n, l, X, ldx, kp, (__nv_bfloat16*)planes,
             (size_t)n * kp, rowexp);
  if (launches) *launches += 2;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

int oz_slice_rows(cudaStream_t st, int n, int l, const double* X, int ldx, double* Xt, int kp, void* planes,
                  int* rowexp, int* launches) {
  if (n <= 0) return 0;
  launch_dep(st, dim3(ceil_div(n, 32), ceil_div(l, 32)), dim3(32, 8), 0, transpose_kernel, n, l, X, ldx, Xt, l);
  // (a thread takes four entries of a row)
  const int threads = std::min(256, std::max(32, ceil_div(kp / 4, 32) * 32));
  launch_dep(st, n, threads, 0, oz_slice_rows_kernel, l, Xt, l, kp, (__nv_bfloat16*)planes, (size_t)n * kp, rowexp);
  if (launches) *launches += 2;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

int oz_slice_cols(cudaStream_t st, int n, int q, const double* Y, int ldy, int kp, void* planes, int* colexp,
                  int* launches) {
  if (q <= 0) return 0;
  launch_dep(st, dim3(q, slice_parts(kp, q)), 256, 0, oz_slice_cols_kernel, n, Y, ldy, kp, (__nv_bfloat16*)planes, (size_t)q * kp, colexp);
  if (launches) ++*launches;
  CHASE_CUDA_TRY(cudaGetLastError());
  return 0;
}

template int oz_stack_V<double>(cudaStream_t, int, int, const double*, int, double*, int, int*);
template int oz_stack_V<z64>(cudaStream_t, int, int, const z64*, int, double*, int, int*);

}  // namespace chase
