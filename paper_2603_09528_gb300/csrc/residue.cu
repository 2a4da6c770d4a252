// Float64 transform GEMMs on the bf16 tensor cores, exact in a residue number
// system: the eigenbasis transforms of the float64 and Ozaki plans (Sec. 2.2.2
// solution steps 2.1, 2.2, 2.4, 2.5; Algorithm 1 steps 1, 3, 7, 9).
//
// Method (Ozaki, Uchino and Imamura, "Ozaki Scheme II", 2025: integer products
// by modular arithmetic and the Chinese remainder theorem).  Every row of an
// operand (the K values one output contracts with) is rounded once to integers
// on its own scale: |X_B| <= 2^bB for a line of the field, |X_A| <= 2^54 for a
// row of the transform matrix.  For pairwise coprime moduli p_1 .. p_n with
// product P, the integer product x = sum_k X_A X_B, |x| < P / 2, is fixed by
// its residues, and each residue is one bf16 GEMM over centred residues
// |r| <= 256 (exact in bf16) with max|r_A| max|r_B| K <= 2^24, so that every
// partial sum is an integer below 2^24 and the float32 accumulator is exact in
// any order.  With  K = 512: 14 moduli below 364 (P > 2^117); K <= 256: 13
// below 514.  Summing slice products instead (Ozaki scheme I, eight 7-bit
// slices, 36 products) needs 2.6 times the tensor-core work for the same 54
// bits.
//
// Reconstruction.  x / P mod 1 = sum_i (r_i y_i mod p_i) / p_i with
// y_i = (P / p_i)^-1 mod p_i; y_i is folded into the matrix's residues, and the
// sum is kept as a 64-bit binary fraction F in registers, whose wrap-around is
// the "mod 1".  Two moduli are taken together: n = r_i p_j + r_j p_i (exact in
// float32), F += n C + rint(n e) with C + e = 2^64 / (p_i p_j).  F is off by at
// most half a unit per pair: 2^-61 P in all, 2^-64.4 P in the root mean square
// (seven pairs).  A typical |x| is ~2^-9.5 P, of which that is 2^-51.5 at most and
// 2^-54.9 typically: the size of one rounding.  The matrix is scaled by P / 2^L (L the bit
// length of P) when it is rounded, so x = F 2^(L-64) times powers of two and the
// result is assembled from its bits: no operation of the float64 pipe (1/64 of
// the float32 rate on GB300) is spent on a point, except the sum of an
// accumulating transform.  The rounding of the operands (2^-54 of a row's
// maximum, not of each value) and that of F are the whole error; the float64 FMA chain it replaces rounds at each
// of the K steps (relative 2-norm error of one transform of noise, K = 512: 9e-17
// against 7.5e-16; K = 64: 9e-17 against 2.6e-16).  In a solve the two cannot be
// told apart element by element either, on grids stretched by 1.5 to 9 and for
// right-hand sides of noise, smooth, with one huge value, or over twelve decades:
// the float64 rounding of the eigenvectors themselves is larger.
//
// Measured (GB300, one transform of 512^3 points): 3.05 ms along x, 3.1 ms along
// y (GEMM 2.0, slicing 1.0 and 1.1), where the float64 FMA GEMM, at that pipe's
// peak, takes 109.7 ms; 256^3 0.30 ms against 6.9.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "cache.h"
#include "ptx.h"
#include "residue.h"
#include "tc.h"
#include "tpt_internal.h"

namespace tpt {
namespace {

size_t al256(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }

constexpr float kMagic = 12582912.0f;           // 1.5 * 2^23: adding it rounds to an integer
constexpr uint32_t kMagicBits = 0x4B400000u;    // its bits; bits(kMagic + n) = kMagicBits + n

// ------------------------------------------------------------------ residues of the operands

// The bits of a row's maximum |x| -> e with max < 2^e (0 for a zero row,
// kRowNonFinite when the row holds an infinity or a NaN).
constexpr int kRowNonFinite = INT_MAX;
__device__ __forceinline__ int row_exponent(unsigned long long maxbits) {
  const int ex = static_cast<int>(maxbits >> 52);
  if (ex == 0x7ff) return kRowNonFinite;
  return ex > 0 ? ex - 1022 : maxbits ? -1010 - __clzll(static_cast<long long>(maxbits)) : 0;
}

// X = round(x 2^(b - e)) for |x| < 2^e, from the bits of x.
__device__ __forceinline__ long long fixed_point(unsigned long long bits, int e, int b) {
  int ex = static_cast<int>((bits >> 52) & 0x7ff);
  unsigned long long mant = bits & ((1ull << 52) - 1);
  if (ex) mant |= 1ull << 52;
  else ex = 1;   // zero or subnormal
  const int sh = 1075 - b + e - ex;   // x = mant 2^(ex - 1075)
  long long X = sh <= 0 ? static_cast<long long>(mant << (-sh & 63))
                        : static_cast<long long>((mant + (1ull << ((sh - 1) & 63))) >> (sh & 63));
  if (sh > 54) X = 0;
  return static_cast<long long>(bits) < 0 ? -X : X;
}

// X, |X| <= 2^57, in balanced base-2^14 digits as floats: X = l0 + 2^14 l1 + 2^28
// l2 + 2^42 l3, |l3| <= 2^15.
__device__ __forceinline__ void limbs(long long X, float (&l)[4]) {
  const unsigned long long Y = static_cast<unsigned long long>(X) + ((1ull << 13) + (1ull << 27) + (1ull << 41));
  const uint32_t lo = static_cast<uint32_t>(Y);
  const uint32_t m1 = static_cast<uint32_t>(Y >> 14) & 0x3fffu;
  const uint32_t m2 = static_cast<uint32_t>(Y >> 28) & 0x3fffu;
  const int top = static_cast<int>(static_cast<long long>(Y) >> 42);
  l[0] = __uint_as_float(0x4B000000u | (lo & 0x3fffu)) - (8388608.0f + 8192.0f);
  l[1] = __uint_as_float(0x4B000000u | m1) - (8388608.0f + 8192.0f);
  l[2] = __uint_as_float(0x4B000000u | m2) - (8388608.0f + 8192.0f);
  l[3] = __uint_as_float(kMagicBits + static_cast<uint32_t>(top)) - kMagic;
}

__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }

// Residues of four values, two neighbouring pairs (limbs l[j] as pairs), for
// every modulus: v = 2^k X mod p up to a multiple of p, from the digits times
// 2^(k + 14 j) mod p (|v| < 2^24, exact), r = v - p rint(v / p), stored as two
// bf16 at dst + i * Kp for modulus i (and dst + 64 + i * Kp for the second pair
// when `two`).  Paired float32 instructions, and the constants of a modulus
// loaded once for both pairs.  The rounded 1/p can take q past a tie for large v:
// |r| is at most data_residue_max(p), p / 2 or one more.
__device__ __forceinline__ void store_residues(const SliceConst& sc, int k, const float2 (&l)[2][4], bool two,
                                               __nv_bfloat16* dst, int Kp) {
  const float2 mg = both(kMagic), nmg = both(-kMagic);
#pragma unroll 2
  for (int i = 0; i < sc.nm; ++i) {
    const float4 c = sc.c[k][i];
    const float inv = sc.inv[i], np = -sc.p[i];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float2 v = __fmul2_rn(l[h][0], both(c.x));
      v = __ffma2_rn(l[h][1], both(c.y), v);
      v = __ffma2_rn(l[h][2], both(c.z), v);
      v = __ffma2_rn(l[h][3], both(c.w), v);
      const float2 q = __fadd2_rn(__ffma2_rn(v, both(inv), mg), nmg);
      const float2 r = __ffma2_rn(q, both(np), v);
      if (h == 0 || two) *reinterpret_cast<__nv_bfloat162*>(dst + 64 * h) = __float22bfloat162_rn(r);
    }
    dst += Kp;
  }
}

// One line of K values (get(k): the bits of value k) by one warp: the row
// exponent, then the residue planes; columns K..Kp-1 are zero.  A non-finite
// line gets zero residues and the exponent kRowNonFinite, which the GEMM's
// epilogue turns into NaN.
template <typename Get>
__device__ __forceinline__ void slice_line(const SliceConst& sc, int K, int Kp, Get get, __nv_bfloat16* dst,
                                           int* expo, int lane) {
  unsigned long long m = 0;
  for (int k = lane; k < K; k += 32) m = max(m, get(k) & 0x7fffffffffffffffull);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int e = row_exponent(m);
  // A line whose values are mostly small against its maximum has a product sum
  // far below K max|X_A| max|X_B|: it is scaled up by the 2^up that its sum of
  // |X_B| leaves free, by finer rounding and then by its residues' scale, so that
  // x keeps the resolution of the fraction F.  t sums an upper bound of
  // |x| / 2^(e - 20), from the leading 20 bits (a subnormal value's are below
  // those of the smallest normal one, which is the bound it gets); a line of
  // subnormal values alone stays as it is.
  const int e1 = e == kRowNonFinite ? 0 : e + 1022;
  uint32_t t = 0;
  for (int k = lane; k < K; k += 32) {
    const uint32_t hi = static_cast<uint32_t>(get(k) >> 32);
    const int d = e1 - static_cast<int>((hi >> 20) & 0x7ff);
    t += d < 20 && d >= 0 ? ((0x100000u | (hi & 0xfffffu)) >> (d + 1)) + 1u : 1u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  int up = sc.L - 35 - sc.bits - (32 - __clz(static_cast<int>(t + 2u)));
  up = up < 0 || e == kRowNonFinite || e1 < 1 ? 0 : up > kMaxUp ? kMaxUp : up;
  if (lane == 0) *expo = e == kRowNonFinite ? e : e - up;
  const int more = min(up, kMaxDataBits - sc.bits);   // as far as the digits reach, the line keeps more bits
  const int bits = sc.bits + more;
  up -= more;
  for (int k = 2 * lane; k < Kp; k += 128) {
    float2 l[2][4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int kh = k + 64 * h;
      long long x0 = 0, x1 = 0;
      if (e != kRowNonFinite) {
        if (kh < K) x0 = fixed_point(get(kh), e, bits);
        if (kh + 1 < K) x1 = fixed_point(get(kh + 1), e, bits);
      }
      float a[4], b[4];
      limbs(x0, a);
      limbs(x1, b);
#pragma unroll
      for (int j = 0; j < 4; ++j) l[h][j] = make_float2(a[j], b[j]);
    }
    store_residues(sc, up, l, k + 64 < Kp, dst + k, Kp);
  }
}

// x lines: line r is K contiguous values at src + r K; one warp per line.
__global__ void __launch_bounds__(256)
slice_x_kernel(long long rows, int K, int Kp, const double* __restrict__ src, __nv_bfloat16* __restrict__ dst,
               int* __restrict__ expo, const __grid_constant__ SliceConst sc) {
  const int lane = threadIdx.x % 32;
  const long long warps = static_cast<long long>(gridDim.x) * (blockDim.x / 32);
  for (long long r = blockIdx.x * static_cast<long long>(blockDim.x / 32) + threadIdx.x / 32; r < rows; r += warps) {
    const unsigned long long* row = reinterpret_cast<const unsigned long long*>(src) + r * K;
    slice_line(sc, K, Kp, [&](int k) { return __ldg(row + k); }, dst + r * (static_cast<long long>(sc.nm) * Kp),
               expo + r, lane);
  }
}

// y lines of a slab of z planes: line (i, k) is the K = ny values at stride nx.
// A block takes LB neighbouring lines of one plane through shared memory (rows
// of LB * 8 bytes in, pitch odd in 8-byte words: no bank conflicts).
template <int LB>
__global__ void __launch_bounds__(256)
slice_y_kernel(int nx, int K, int Kp, const double* __restrict__ src, __nv_bfloat16* __restrict__ dst,
               int* __restrict__ expo, const __grid_constant__ SliceConst sc) {
  extern __shared__ unsigned long long tile[];
  const int pitch = K | 1;
  const int tiles = (nx + LB - 1) / LB;
  const long long plane = blockIdx.x / tiles;
  const int i0 = static_cast<int>(blockIdx.x % tiles) * LB;
  const unsigned long long* in = reinterpret_cast<const unsigned long long*>(src) + plane * nx * K;
#pragma unroll 8
  for (int t = threadIdx.x; t < LB * K; t += 256) {
    const int i = t % LB, j = t / LB;
    if (i0 + i < nx) tile[i * pitch + j] = __ldg(in + i0 + i + static_cast<long long>(nx) * j);
  }
  __syncthreads();
  const int lane = threadIdx.x % 32;
  for (int i = threadIdx.x / 32; i < LB && i0 + i < nx; i += 8) {
    const unsigned long long* row = tile + i * pitch;
    const long long r = plane * nx + i0 + i;
    slice_line(sc, K, Kp, [&](int k) { return row[k]; }, dst + r * (static_cast<long long>(sc.nm) * Kp), expo + r,
               lane);
  }
}

// Rows of a float64 transform matrix on the device: element (r, k) at
// src[r rs + k cs].
struct DenseRows {
  const double* src;
  long long rs, cs;
  __device__ __forceinline__ double operator()(int r, int k) const { return src[r * rs + k * cs]; }
};

// Rows of the real DFT (kind 0, half-complex mode order) or DCT-II (kind 1) of n
// points, a power of two, or of their exact inverses; tab holds cos(2 pi m / n)
// and sin(2 pi m / n), m < n, or cos(2 pi m / 4n), m < 4n.
struct FourierRows {
  const double* tab;
  int n, kind, inverse;
  __device__ __forceinline__ double operator()(int r, int k) const {
    const int mode = inverse ? k : r, point = inverse ? r : k;
    double v;
    if (kind == 1) {
      v = tab[static_cast<int>(static_cast<long long>(mode) * (2 * point + 1) & (4 * n - 1))];
    } else if (mode == 0) {
      v = 1.0;
    } else if (mode == n - 1) {
      v = point % 2 ? -1.0 : 1.0;
    } else {
      const int m = static_cast<int>(static_cast<long long>((mode + 1) / 2) * point & (n - 1));
      v = mode % 2 ? tab[m] : tab[n + m];
    }
    if (inverse) v *= (mode == 0 || (kind == 0 && mode == n - 1) ? 1.0 : 2.0) / n;
    return v;
  }
};

// Transform-matrix table: row r of K values rounded to X_A = round(a 2^(54 - e)
// G / 2^64) and stored as the residues of X_A y_i; one block per row.
template <typename Rows>
__global__ void __launch_bounds__(256)
matrix_residues_kernel(int K, int Kp, const Rows rows, __nv_bfloat16* __restrict__ dst,
                       int* __restrict__ expo, const __grid_constant__ MatrixConst mc) {
  __shared__ unsigned long long wmax[8];
  const long long r = blockIdx.x;
  auto get = [&](int k) {
    return static_cast<unsigned long long>(__double_as_longlong(rows(static_cast<int>(r), k)));
  };
  unsigned long long m = 0;
  for (int k = threadIdx.x; k < K; k += blockDim.x) m = max(m, get(k) & 0x7fffffffffffffffull);
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (threadIdx.x % 32 == 0) wmax[threadIdx.x / 32] = m;
  __syncthreads();
  for (int w = 0; w < 8; ++w) m = max(m, wmax[w]);
  const int e = row_exponent(m);
  if (threadIdx.x == 0) expo[r] = e;
  for (int k = threadIdx.x; k < Kp; k += blockDim.x) {
    long long X = 0;
    if (k < K && e != kRowNonFinite) {
      const unsigned long long bits = get(k);
      const int ex = static_cast<int>((bits >> 52) & 0x7ff);
      if (ex != 0) {
        const unsigned long long mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
        const unsigned long long hi = __umul64hi(mant, mc.scale), lo = mant * mc.scale;
        const int sh = 64 + 1075 - kMatrixBits + e - ex;   // >= 63: mant < 2^53, X <= 2^kMatrixBits
        if (sh == 63) {
          X = static_cast<long long>((hi << 1) | (lo >> 63)) + static_cast<long long>((lo >> 62) & 1);
        } else if (sh == 64) {
          X = static_cast<long long>(hi + (lo >> 63));
        } else if (sh < 64 + 54) {
          X = static_cast<long long>((hi + (1ull << (sh - 65))) >> (sh - 64));
        }
        if (bits >> 63) X = -X;
      }
    }
    for (int i = 0; i < mc.nm; ++i) {
      const int p = mc.p[i];
      int v = static_cast<int>(X % p) * mc.y[i] % p;   // |v| < p
      if (2 * v > p) v -= p;
      if (2 * v < -p) v += p;
      dst[(r * mc.nm + i) * Kp + k] = __float2bfloat16_rn(static_cast<float>(v));
    }
  }
}

// ------------------------------------------------------------------ the GEMM

constexpr int BM = 128, BK = 64;
constexpr int kBufs = 4;                       // tensor-memory accumulators of BN columns
constexpr int kEpiWarps = 16;
constexpr int kThreads = 32 * (2 + kEpiWarps);
template <int BN>
struct RCfg {
  static constexpr int kABytes = BM * BK * 2, kStage = kABytes + BN * BK * 2;
  static constexpr int kStages = 192 * 1024 / kStage;
  static constexpr int kCols = 4 * BN / kEpiWarps;   // columns of an epilogue thread
  static constexpr int kSmem = kStages * kStage + 1024 /* alignment */ + 384 /* barriers, left */;
};

// 2^k times the 64-bit integer F, rounded to nearest even
__device__ __forceinline__ double assemble(long long F, int k) {
  if (F == 0) return 0.0;
  const unsigned long long a = F < 0 ? 0ull - static_cast<unsigned long long>(F) : static_cast<unsigned long long>(F);
  const int lz = __clzll(static_cast<long long>(a));
  const unsigned long long m = a << lz;
  unsigned long long top = m >> 11;
  const uint32_t rem = static_cast<uint32_t>(m) & 0x7ffu;
  top += (rem + (static_cast<uint32_t>(top) & 1u) > 0x400u) ? 1u : 0u;
  const int ex = 1085 - lz + k;                // exponent field less the hidden bit of top
  if (ex < 0 || ex > 2044) {                   // subnormal or overflowing results
    const double v = scalbn(static_cast<double>(top), 11 - lz + k);
    return F < 0 ? -v : v;
  }
  unsigned long long bits = (static_cast<unsigned long long>(ex) << 52) + top;
  if (F < 0) bits |= 1ull << 63;
  return __longlong_as_double(static_cast<long long>(bits));
}

// D = A B^T through the residues of A (M rows) and B (N rows): persistent, one
// CTA per SM, tiles of 128 x BN; for each tile the moduli in turn, each one
// K = Kp bf16 product into its own tensor-memory accumulator (four of them:
// two pairs, so the tensor cores run ahead while the epilogue folds a pair).
//   warp 0     TMA producer (128-byte rows, 128-byte swizzle, 192 KB of stages)
//   warp 1     tcgen05.mma issue; padding K steps of the last chunk are skipped
//   warps 2-17 epilogue: a warp owns 32 rows x BN / 4 columns, one 64-bit fraction
//              per element in registers over all moduli (sixteen warps: four a
//              scheduler, and half the unrolled code of eight)
// Element (m, n) is written (or added) at (m % rm) + (m / rm) sm + n sn.  Every
// wait is bounded; a timeout sets bits in *err, and the CTA drains and exits with
// NaN in the tiles that it has not finished, as do the CTAs that find the flag
// set, so that no later kernel or caller takes stale memory for a result.
// DROP: failure-detection test; the producer issues no loads, the waits are short.
template <int BN, bool DROP = false>
__global__ void __launch_bounds__(kThreads, 1)
residue_gemm_kernel(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB,
                    const __grid_constant__ ResidueGemm g) {
  constexpr int kABytes = RCfg<BN>::kABytes, kStage = RCfg<BN>::kStage, kStages = RCfg<BN>::kStages;
  constexpr int kCols = RCfg<BN>::kCols;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * kStage);
  uint64_t* accf = bars + 2 * kStages;          // accumulator full
  uint64_t* acce = accf + kBufs;                // accumulator drained
  uint64_t* mdone = acce + kBufs;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mdone + 1);
  long long* left = reinterpret_cast<long long*>(mdone + 2);   // an epilogue warp's first unfinished tile
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int num_m = (g.M + BM - 1) / BM, num_n = (g.N + BN - 1) / BN;
  const long long tiles = static_cast<long long>(num_m) * num_n;
  const int nk = g.Kp / BK;
  constexpr uint32_t polls = DROP ? 1u << 10 : 1u << 22;
  // A timed-out CTA stops by its own bounded waits; the others look at the flag
  // once a tile, with the load in flight over the tile before (a load per ring
  // stage put ~700 cycles into the producer's loop).
  auto aborted = [&]() -> int { return g.err ? *reinterpret_cast<volatile int*>(g.err) : 0; };
  auto origin = [&](long long q, int& m0, int& n0) {
    const long long f = g.n_fastest ? num_n : num_m;
    const int lo = static_cast<int>(q % f), hi = static_cast<int>(q / f);
    m0 = (g.n_fastest ? hi : lo) * BM;
    n0 = (g.n_fastest ? lo : hi) * BN;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      ptx::mbar_init(ptx::smem_u32(&bars[s]), 1);
      ptx::mbar_init(ptx::smem_u32(&bars[kStages + s]), 1);
    }
    for (int b = 0; b < kBufs; ++b) {
      ptx::mbar_init(ptx::smem_u32(&accf[b]), 1);
      ptx::mbar_init(ptx::smem_u32(&acce[b]), kEpiWarps);
    }
    ptx::mbar_init(ptx::smem_u32(mdone), 1);
    ptx::fence_mbar_init();
    for (int w = 0; w < kEpiWarps; ++w) left[w] = tiles;
  }
  if (warp == 1) {
    ptx::tmem_alloc(ptx::smem_u32(tmem_slot), kBufs * BN);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    ptx::prefetch_tmap(&tA);
    ptx::prefetch_tmap(&tB);
    bool ok = true;
    long long it = 0;
    int stop = 0;
    for (long long q = blockIdx.x; q < tiles && ok && !stop; q += gridDim.x) {
      int m0, n0;
      origin(q, m0, n0);
      stop = aborted();
      for (int c = 0; c < g.nm * nk; ++c, ++it) {   // chunk c: modulus c / nk, K offset (c % nk) * 64
        const int s = static_cast<int>(it % kStages);
        const long long round = it / kStages;
        if (round > 0)
          ok = ptx::mbar_wait(ptx::smem_u32(&bars[kStages + s]), static_cast<uint32_t>((round - 1) & 1), g.err,
                              ptx::kErrWaitEmpty, polls);
        if (DROP) ok = false;
        if (!ok) break;
        uint8_t* st = smem + s * kStage;
        const uint32_t full = ptx::smem_u32(&bars[s]);
        ptx::mbar_arrive_expect_tx(full, kStage);
        ptx::tma_load_2d(ptx::smem_u32(st), &tA, full, c * BK, m0);
        ptx::tma_load_2d(ptx::smem_u32(st + kABytes), &tB, full, c * BK, n0);
      }
    }
    const long long first = it > kStages ? it - kStages : 0;
    for (long long k = first; k < it; ++k)   // every issued copy has landed before the CTA may exit
      ptx::mbar_wait(ptx::smem_u32(&bars[k % kStages]), static_cast<uint32_t>((k / kStages) & 1), g.err,
                     ptx::kErrWaitDrain, polls);
  } else if (warp == 1) {
    // The whole warp runs the loop and one elected lane issues: descriptors and
    // barrier addresses stay in uniform registers (a lone thread building them
    // took ~170 cycles per MMA, more than twice the MMA itself).
    constexpr uint32_t idesc = ptx::instr_desc(1u, BM, BN);
    const uint32_t issue = ptx::elect_one();
    const uint64_t desc0 = ptx::smem_desc_k_sw128(ptx::smem_u32(smem));
    const uint32_t bar0 = ptx::smem_u32(bars);
    const int last = (g.K - (nk - 1) * BK + 15) / 16;   // K steps of the last chunk
    bool ok = true;
    uint32_t s = 0, par = 0, b = 0, bpar = 1, first = 1;   // ring stage and its parity; accumulator
    int stop = 0;
    for (long long q = blockIdx.x; q < tiles && ok; q += gridDim.x) {
      if (__any_sync(0xffffffffu, stop)) break;
      stop = aborted();
      for (int i = 0; i < g.nm && ok; ++i) {
        if (!first)
          ok = ptx::mbar_wait_warp(bar0 + 8 * (2 * kStages + kBufs + b), bpar, g.err, ptx::kErrWaitAccum, polls);
        if (!ok) break;
        ptx::tc_fence_after();
        const uint32_t d = tmem + b * BN;
        for (int kc = 0; kc < nk; ++kc) {
          ok = ptx::mbar_wait_warp(bar0 + 8 * s, par, g.err, ptx::kErrWaitFull, polls);
          if (!ok) break;
          ptx::tc_fence_after();
          const uint64_t da = desc0 + s * (kStage >> 4), db = da + (kABytes >> 4);
          const int steps = kc == nk - 1 ? last : BK / 16;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            if (kk < steps) ptx::mma_bf16_if(issue, d, da + 2 * kk, db + 2 * kk, idesc, (kc > 0 || kk > 0) ? 1u : 0u);
          ptx::mma_commit_if(issue, bar0 + 8 * (kStages + s));
          if (++s == kStages) {
            s = 0;
            par ^= 1;
          }
        }
        ptx::mma_commit_if(issue, bar0 + 8 * (2 * kStages + b));
        if (++b == kBufs) {
          b = 0;
          bpar ^= 1;
          first = 0;
        }
      }
    }
    // every MMA has completed before the tensor memory is freed
    ptx::mma_commit_if(issue, ptx::smem_u32(mdone));
    ptx::mbar_wait_warp(ptx::smem_u32(mdone), 0u, g.err, ptx::kErrWaitDrain, polls);
  } else if (warp >= 2) {
    const int quarter = warp % 4;                // tensor-memory lanes 32 * quarter ..
    const int col0 = ((warp - 2) / 4) * kCols;
    const float2 mg = both(kMagic), nmg = both(-kMagic);
    long long t = 0;
    bool go = true;
    int stop = 0;
    for (long long q = blockIdx.x; q < tiles; q += gridDim.x) {
      int m0, n0;
      origin(q, m0, n0);
      if (__any_sync(0xffffffffu, stop)) {        // tcgen05.ld is warp-collective
        if (lane == 0) left[warp - 2] = q;
        break;
      }
      stop = aborted();
      long long F[kCols];
#pragma unroll
      for (int c = 0; c < kCols; ++c) F[c] = g.f0;
      for (int j = 0; j < g.npair; ++j) {
        const ResiduePair& pr = g.pair[j];
        const bool two = 2 * j + 1 < g.nm;
        const int b0 = static_cast<int>(t % kBufs), b1 = static_cast<int>((t + 1) % kBufs);
        bool ok = ptx::mbar_wait(ptx::smem_u32(&accf[b0]), static_cast<uint32_t>((t / kBufs) & 1), g.err,
                                 ptx::kErrWaitAccum, polls);
        if (two && ok)
          ok = ptx::mbar_wait(ptx::smem_u32(&accf[b1]), static_cast<uint32_t>(((t + 1) / kBufs) & 1), g.err,
                              ptx::kErrWaitAccum, polls);
        ptx::tc_fence_after();
        if (!__all_sync(0xffffffffu, ok)) {
          go = false;
          break;
        }
        const uint32_t base = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + static_cast<uint32_t>(col0);
#pragma unroll
        for (int c0 = 0; c0 < kCols; c0 += 8) {
          uint32_t s1[8], s2[8];
          ptx::tmem_ld_32x32b_x8(base + static_cast<uint32_t>(b0 * BN + c0), s1);
          ptx::tmem_ld_32x32b_x8(base + static_cast<uint32_t>((two ? b1 : b0) * BN + c0), s2);
          ptx::tmem_ld_wait();
#pragma unroll
          for (int c = 0; c < 8; c += 2) {
            const float2 a = make_float2(__uint_as_float(s1[c]), __uint_as_float(s1[c + 1]));
            const float2 b = make_float2(__uint_as_float(s2[c]), __uint_as_float(s2[c + 1]));
            const float2 qa = __fadd2_rn(__ffma2_rn(a, both(pr.inv1), mg), nmg);
            const float2 qb = __fadd2_rn(__ffma2_rn(b, both(pr.inv2), mg), nmg);
            const float2 ra = __ffma2_rn(qa, both(-pr.p1), a);
            const float2 rb = __ffma2_rn(qb, both(-pr.p2), b);
            const float2 n = __ffma2_rn(ra, both(pr.f1), __fmul2_rn(rb, both(pr.f2)));
            const float2 u = __fadd2_rn(n, mg);
            const float2 v = __ffma2_rn(n, both(pr.e), mg);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int ui = __float_as_int(h ? u.y : u.x);
              const uint32_t vi = __float_as_uint(h ? v.y : v.x);
              const unsigned long long w =
                  static_cast<unsigned long long>(static_cast<long long>(ui) * pr.clo) + F[c0 + c + h];
              const unsigned long long wh = static_cast<uint32_t>(ui) * static_cast<uint32_t>(pr.chi);   // mod 2^32
              F[c0 + c + h] = static_cast<long long>(w + (wh << 32) + vi);
            }
          }
        }
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) {
          ptx::mbar_arrive(ptx::smem_u32(&acce[b0]));
          if (two) ptx::mbar_arrive(ptx::smem_u32(&acce[b1]));
        }
        t += two ? 2 : 1;
      }
      if (!go) {
        if (lane == 0) left[warp - 2] = q;
        break;
      }
      const int m = m0 + quarter * 32 + lane;
      if (m < g.M) {
        const int ea = g.expA[m];
        double* out = g.out + (m % g.rm) + static_cast<long long>(m / g.rm) * g.sm;
#pragma unroll
        for (int c = 0; c < kCols; ++c) {
          const int n = n0 + col0 + c;
          if (n < g.N) {
            const int eb = __ldg(g.expB + n);
            double v = (ea == kRowNonFinite || eb == kRowNonFinite) ? __longlong_as_double(0x7ff8000000000000ll)
                                                                    : assemble(F[c], ea + eb + g.shift);
            double* o = out + static_cast<long long>(n) * g.sn;
            if (g.accumulate) v += *o;
            *o = v;
          }
        }
      }
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) ptx::tmem_dealloc(tmem, kBufs * BN);
  // tiles given up after a timeout (here, where the epilogue's registers are free)
  if (warp < 2) return;
#pragma unroll 1
  for (long long q = left[warp - 2]; q < tiles; q += gridDim.x) {
    int m0, n0;
    origin(q, m0, n0);
    const int m = m0 + (warp % 4) * 32 + lane, n1 = n0 + ((warp - 2) / 4) * kCols;
    if (m >= g.M) continue;
    double* out = g.out + (m % g.rm) + static_cast<long long>(m / g.rm) * g.sm;
#pragma unroll 1
    for (int n = n1; n < min(g.N, n1 + kCols); ++n)
      out[static_cast<long long>(n) * g.sn] = __longlong_as_double(0x7ff8000000000000ll);
  }
}

// ------------------------------------------------------------------ host side

int gcd(int a, int b) { return b ? gcd(b, a % b) : a; }

// The inverse of a modulo p (coprime), 1 <= result < p (p is small).
int inverse_mod(int a, int p) {
  for (int x = 1; x < p; ++x)
    if (static_cast<long long>(a) * x % p == 1) return x;
  return 1;   // p == 1
}

// 2^bit mod p, centred.
int centred_power(int bit, int p) {
  const int v = static_cast<int>((1LL << bit) % p);
  return 2 * v > p ? v - p : v;
}

// Largest |r| that store_residues leaves for modulus p: r = v - p rint(v inv) with
// inv = (1 + d) / p, so |r| <= p / 2 + |v| |d|, |v| at most the digits' largest
// magnitudes (2^13 three times and 2^15) times their constants'.
int data_residue_max(int p) {
  long long vmax = 0;
  for (int k = 0; k <= kMaxUp; ++k) {
    long long v = 0;
    for (int j = 0; j < 4; ++j) v += (j < 3 ? 1LL << 13 : 1LL << 15) * std::abs(centred_power(k + 14 * j, p));
    vmax = std::max(vmax, v);
  }
  const double d = static_cast<double>(1.0f / p) * p - 1.0;   // exact
  return static_cast<int>(0.5 * p + static_cast<double>(vmax) * std::fabs(d));
}

}  // namespace

bool residue_system(int K, ResidueSystem* s) {
  if (K < 1 || K > kResidueMaxK) return false;
  int rmax = 1;
  while (rmax < 256 && static_cast<long long>(rmax + 1) * (rmax + 1) * K <= (1LL << 24)) ++rmax;
  int lk = 0;
  while ((1 << lk) < K) ++lk;
  std::memset(s, 0, sizeof(*s));
  unsigned __int128 P = 1;
  for (int p = 2 * rmax + 1; p > 2; --p) {
    if (p % 2 == 0 && p / 2 > rmax) continue;
    bool coprime = true;
    for (int i = 0; i < s->nm; ++i) coprime = coprime && gcd(p, s->p[i]) == 1;
    if (!coprime) continue;
    // exact operands and sums, proven for this modulus (a residue one beyond p / 2
    // is too much for p = 495 at K = 274 and p = 491 at K = 279 only)
    const long long rdata = data_residue_max(p);
    if (rdata > 256 || rdata * (p / 2) * K > (1LL << 24)) continue;
    s->p[s->nm++] = p;
    P *= static_cast<unsigned>(p);
    int L = 0;
    while (L < 128 && (P >> L) != 0) ++L;
    // |x| <= K 2^bB (2^54 P / 2^L + 1/2) must stay below P / 2
    const int bits = L - 2 - kMatrixBits - lk;
    if (bits >= kDataBits) {
      s->L = L;
      s->bits = bits < kMaxDataBits ? bits : kMaxDataBits;
      break;
    }
    if (s->nm == kMaxModuli) return false;
  }
  if (s->L == 0) return false;
  s->scale = static_cast<unsigned long long>((P << (128 - s->L)) >> 64);
  for (int i = 0; i < s->nm; ++i) {
    int rest = 1;
    for (int j = 0; j < s->nm; ++j)
      if (j != i) rest = static_cast<int>(static_cast<long long>(rest) * s->p[j] % s->p[i]);
    s->y[i] = inverse_mod(rest % s->p[i], s->p[i]);
  }
  return true;
}

namespace {

SliceConst slice_const(const ResidueSystem& s) {
  SliceConst c;
  std::memset(&c, 0, sizeof(c));
  c.nm = s.nm;
  c.bits = s.bits;
  c.L = s.L;
  for (int i = 0; i < s.nm; ++i) {
    const int p = s.p[i];
    auto centred = [&](int bit) { return static_cast<float>(centred_power(bit, p)); };
    for (int k = 0; k <= kMaxUp; ++k)
      c.c[k][i] = make_float4(centred(k), centred(k + 14), centred(k + 28), centred(k + 42));
    c.inv[i] = 1.0f / p;
    c.p[i] = static_cast<float>(p);
  }
  return c;
}

void gemm_const(const ResidueSystem& s, ResidueGemm* g) {
  g->nm = s.nm;
  g->npair = (s.nm + 1) / 2;
  unsigned long long f0 = 0;
  for (int j = 0; j < g->npair; ++j) {
    const int p1 = s.p[2 * j], p2 = 2 * j + 1 < s.nm ? s.p[2 * j + 1] : 1;
    const int pp = p1 * p2;
    const unsigned __int128 one = static_cast<unsigned __int128>(1) << 64;
    const unsigned long long q = static_cast<unsigned long long>(one / pp);        // < 2^56
    const int rem = static_cast<int>(one % pp);
    // 2^64 / pp = C + e with |e| <= 1/2; C = chi 2^32 + clo, clo signed
    const unsigned long long C = 2 * rem > pp ? q + 1 : q;
    ResiduePair& pr = g->pair[j];
    pr.e = static_cast<float>((2LL * rem > pp ? rem - pp : rem) / static_cast<double>(pp));
    pr.clo = static_cast<int>(static_cast<uint32_t>(C));
    pr.chi = static_cast<int>((C - static_cast<unsigned long long>(static_cast<long long>(pr.clo))) >> 32);
    pr.p1 = static_cast<float>(p1);
    pr.p2 = static_cast<float>(p2);
    pr.inv1 = 1.0f / p1;
    pr.inv2 = 1.0f / p2;
    pr.f1 = static_cast<float>(p2);
    pr.f2 = p2 == 1 ? 0.0f : static_cast<float>(p1);   // a lone modulus: its pair's accumulator does not count
    f0 -= kMagicBits * C + kMagicBits;   // the magic offsets of u and v
  }
  g->f0 = static_cast<long long>(f0);
  g->shift = s.L - 64 - kMatrixBits - s.bits;
}

// Columns of a tile: rounds of tiles over the SMs times (columns + 70).  A tile's
// epilogue takes 0.14 us a column, its start and the moduli's turns ~10 us, so
// small transforms, which do not fill the chip with 128-column tiles, spread
// their columns over more CTAs (32^3 22 -> 9.4 us, 61x97x75 30 -> 13).
int tile_columns(int M, int N, int sms) {
  int best = 128;
  long long cost = -1;
  for (int bn = 128; bn >= 32; bn /= 2) {
    const long long tiles = static_cast<long long>((M + BM - 1) / BM) * ((N + bn - 1) / bn);
    const long long c = (tiles + sms - 1) / sms * (bn + 70);
    if (cost < 0 || c < cost) {
      cost = c;
      best = bn;
    }
  }
  return best;
}

template <int BN, bool DROP = false>
cudaError_t launch_gemm(const CUtensorMap& a, const CUtensorMap& b, const ResidueGemm& g, int sms, cudaStream_t s) {
  const cudaError_t e = cudaFuncSetAttribute(residue_gemm_kernel<BN, DROP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             RCfg<BN>::kSmem);
  if (e != cudaSuccess) return e;
  const long long tiles = static_cast<long long>((g.M + BM - 1) / BM) * ((g.N + BN - 1) / BN);
  residue_gemm_kernel<BN, DROP>
      <<<static_cast<unsigned>(tiles < sms ? tiles : sms), kThreads, RCfg<BN>::kSmem, s>>>(a, b, g);
  return cudaGetLastError();
}

// Lines of direction d that one pass slices and multiplies (the scratch holds
// their residues): all of them when they fit in the plan's res_cap, else whole
// z planes.
long long lines_per_pass(const tpt_plan_s* p, int d) {
  const ResidueDir& rd = p->res[d];
  const long long per_plane = d == 0 ? p->n[1] : p->n[0];
  const size_t line = static_cast<size_t>(rd.sys.nm) * rd.kp * 2 + sizeof(int);
  long long planes = static_cast<long long>(p->res_cap / (line * static_cast<size_t>(per_plane)));
  if (planes < 1) planes = 1;
  if (planes > p->n[2]) planes = p->n[2];
  return planes * per_plane;
}

}  // namespace

int residue_tables(DevArena& a, int n, const DevDir& dd, int role, bool fft, int kind, ResidueDir* out) {
  ResidueDir rd;
  if (!residue_system(n, &rd.sys)) return TPT_ERR_UNSUPPORTED;
  rd.kp = (n + BK - 1) / BK * BK;
  const size_t tab = al256(static_cast<size_t>(n) * rd.sys.nm * rd.kp * 2), expo = al256(n * sizeof(int));
  MatrixConst mc;
  std::memset(&mc, 0, sizeof(mc));
  mc.nm = rd.sys.nm;
  mc.scale = rd.sys.scale;
  for (int i = 0; i < rd.sys.nm; ++i) {
    mc.p[i] = rd.sys.p[i];
    mc.y[i] = rd.sys.y[i];
  }
  std::vector<double> angles;   // of a Fourier-transformed direction
  if (fft) {
    const long double pi2 = 6.283185307179586476925286766559005768L;
    const int m = kind == 1 ? 4 * n : n;
    for (int k = 0; k < m; ++k) angles.push_back(static_cast<double>(std::cos(pi2 * k / m)));
    if (kind == 0)
      for (int k = 0; k < n; ++k) angles.push_back(static_cast<double>(std::sin(pi2 * k / n)));
  }
  void* mem = nullptr;
  const int st = a.alloc(2 * (tab + expo) + angles.size() * sizeof(double), &mem);
  if (st != TPT_OK) return st;
  char* w = static_cast<char*>(mem);
  double* angles_d = reinterpret_cast<double*>(w + 2 * (tab + expo));
  if (fft && cudaMemcpyAsync(angles_d, angles.data(), angles.size() * sizeof(double), cudaMemcpyHostToDevice,
                             a.stream) != cudaSuccess)
    return TPT_ERR_CUDA;
  for (int inv = 0; inv < 2; ++inv) {
    rd.tab[inv] = w + inv * (tab + expo);
    rd.expo[inv] = reinterpret_cast<int*>(w + inv * (tab + expo) + tab);
    __nv_bfloat16* t = static_cast<__nv_bfloat16*>(rd.tab[inv]);
    note_launch(1);
    if (fft) {
      const FourierRows rows{angles_d, n, kind, inv};
      matrix_residues_kernel<<<n, 256, 0, a.stream>>>(n, rd.kp, rows, t, rd.expo[inv], mc);
    } else {
      // rows = output modes: x transforms read A[r][k] = mat[r + n k], y
      // transforms B[r][k] = mat[k + n r]
      const DenseRows rows{inv ? dd.inv : dd.fwd, role == 0 ? 1 : n, role == 0 ? n : 1};
      matrix_residues_kernel<<<n, 256, 0, a.stream>>>(n, rd.kp, rows, t, rd.expo[inv], mc);
    }
    if (cudaGetLastError() != cudaSuccess) return TPT_ERR_CUDA;
  }
  if (cudaStreamSynchronize(a.stream) != cudaSuccess) return TPT_ERR_CUDA;   // angles dies here; entries are shared
  rd.ready = true;
  *out = rd;
  return TPT_OK;
}

int residue_setup(tpt_plan_s* p, int d) {
  const bool fft = p->xform[d] == TPT_XFORM_FFT;
  if (p->basis[d]) return entry_residue_tables(*p->basis[d], p->ddir[d], d, &p->res[d]);
  return residue_tables(p->arena, p->n[d], p->ddir[d], d, fft, p->fft[d].kind, &p->res[d]);
}

size_t residue_scratch_bytes(const tpt_plan_s* p) {
  size_t most = 0;
  for (int d = 0; d < 2; ++d) {
    if (!p->res[d].ready) continue;
    const size_t lines = static_cast<size_t>(lines_per_pass(p, d));
    const size_t b = al256(lines * p->res[d].sys.nm * p->res[d].kp * 2) + al256(lines * sizeof(int));
    if (b > most) most = b;
  }
  return most;
}

void residue_limit(tpt_plan_s* p, size_t bytes) {
  if (bytes >= residue_scratch_bytes(p)) return;
  p->res_cap = bytes;   // lines_per_pass leaves out the alignment of its two regions:
  if (residue_scratch_bytes(p) > bytes && bytes > 512) p->res_cap = bytes - 512;
  if (residue_scratch_bytes(p) > bytes && !p->ozaki) p->res[0].ready = p->res[1].ready = false;
  ++p->generation;      // recorded graphs hold the old passes
}

cudaError_t residue_transform(const tpt_plan_s* p, int d, bool inverse, const double* in, double* out,
                              bool accumulate, void* scratch, int* err, cudaStream_t s) {
  const int nx = p->n[0], ny = p->n[1], nz = p->n[2];
  const ResidueDir& rd = p->res[d];
  const int n = p->n[d], kp = rd.kp, ld = rd.sys.nm * kp;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->dev);
  const long long per_pass = lines_per_pass(p, d);
  const long long per_plane = d == 0 ? ny : nx, total = per_plane * nz, slab = static_cast<long long>(nx) * ny;
  __nv_bfloat16* sl = static_cast<__nv_bfloat16*>(scratch);
  int* expo = reinterpret_cast<int*>(static_cast<char*>(scratch) + al256(static_cast<size_t>(per_pass) * ld * 2));
  const SliceConst sc = slice_const(rd.sys);
  ResidueGemm g;
  std::memset(&g, 0, sizeof(g));
  gemm_const(rd.sys, &g);
  g.K = n;
  g.Kp = kp;
  g.err = err;
  g.accumulate = accumulate ? 1 : 0;
  CUtensorMap mat, data;
  const int tab = inverse ? 1 : 0;
  cudaError_t e = cudaSuccess;
  for (long long l0 = 0; l0 < total; l0 += per_pass) {
    const int lines = static_cast<int>(total - l0 < per_pass ? total - l0 : per_pass);
    const long long off = l0 / per_plane * slab;   // first z plane of the pass
    note_launch(2);
    if (d == 0) {
      const long long blocks = (lines + 7) / 8;
      slice_x_kernel<<<static_cast<unsigned>(blocks < 16LL * sms ? blocks : 16LL * sms), 256, 0, s>>>(
          lines, n, kp, in + off, sl, expo, sc);
    } else {
      const unsigned planes = static_cast<unsigned>(lines / nx);
      auto run = [&](auto kern, int lb) -> cudaError_t {
        const int bytes = lb * (n | 1) * 8;
        const cudaError_t ea = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 16 * 1025 * 8);
        if (ea != cudaSuccess) return ea;
        kern<<<planes * static_cast<unsigned>((nx + lb - 1) / lb), 256, bytes, s>>>(nx, n, kp, in + off, sl, expo,
                                                                                     sc);
        return cudaGetLastError();
      };
      e = n <= 1024 ? run(slice_y_kernel<16>, 16) : run(slice_y_kernel<8>, 8);
      if (e != cudaSuccess) return e;
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    g.out = out + off;
    g.sn = nx;
    if (d == 0) {   // the matrix's rows are the output's x index
      g.M = nx;
      g.N = lines;
      g.rm = nx;
      g.sm = 0;
      g.expA = rd.expo[tab];
      g.expB = expo;
      g.n_fastest = 0;
    } else {
      g.M = lines;
      g.N = ny;
      g.rm = nx;
      g.sm = slab;
      g.expA = expo;
      g.expB = rd.expo[tab];
      g.n_fastest = 1;
    }
    const int bn = p->res_drop_loads ? 128 : tile_columns(g.M, g.N, sms);
    if (!tc::make_operand_map(&mat, rd.tab[tab], n, ld, ld, d == 0 ? BM : bn)) return cudaErrorInvalidValue;
    if (!tc::make_operand_map(&data, sl, lines, ld, ld, d == 0 ? bn : BM)) return cudaErrorInvalidValue;
    const CUtensorMap& ma = d == 0 ? mat : data;
    const CUtensorMap& mb = d == 0 ? data : mat;
    e = p->res_drop_loads ? launch_gemm<128, true>(ma, mb, g, sms, s)
        : bn == 128 ? launch_gemm<128>(ma, mb, g, sms, s) : bn == 64 ? launch_gemm<64>(ma, mb, g, sms, s)
                                                                   : launch_gemm<32>(ma, mb, g, sms, s);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace tpt
