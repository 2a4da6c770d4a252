// float64 kernels of the solve: the eigenbasis-transform GEMM (Sec. 2.2.2,
// Eq. forward-xy / inverse-xy; lines stacked as one GEMM), the modal Thomas
// sweep along z (solution step 2.3, with the gauge of Sec. 3), and the
// 7-point residual r = f - (alpha I + beta L) phi (Sec. 4.1).
//
// float64 arithmetic on GB300 runs at about 1 TFLOP/s (FMA and DMMA alike), so
// these kernels are bound by the float64 pipe, not by HBM; the layouts below
// keep every global access coalesced so that the float64 units stay fed.
#include <cuda_runtime.h>

#include <cmath>
#include <type_traits>

#include "df.h"
#include "tpt_internal.h"

namespace tpt {
namespace {

constexpr int TM = 64, TN = 64, TK = 16;   // block tile and k-step
constexpr int TX = 16, TY = 16;            // 256 threads, 4 x 4 outputs each

// C_b = A_b B_b (+ C_b): column-major, ragged edges zero-filled in shared memory.
__global__ void __launch_bounds__(TX * TY)
dgemm_cm_kernel(int M, int N, int K, const double* __restrict__ A, int lda, long long sA,
                const double* __restrict__ B, int ldb, long long sB, double* __restrict__ C,
                int ldc, long long sC, int accumulate) {
  __shared__ double As[TK][TM + 1];
  __shared__ double Bs[TK][TN + 1];
  const int tx = threadIdx.x, ty = threadIdx.y, tid = ty * TX + tx;
  const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
  const long long b = blockIdx.z;
  A += b * sA;
  B += b * sB;
  C += b * sC;
  double acc[4][4];
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0.0;

  for (int k0 = 0; k0 < K; k0 += TK) {
#pragma unroll
    for (int r = 0; r < (TM * TK) / (TX * TY); ++r) {   // A tile, coalesced along m
      const int e = tid + r * TX * TY, m = e % TM, k = e / TM;
      const int gm = m0 + m, gk = k0 + k;
      As[k][m] = (gm < M && gk < K) ? A[gm + static_cast<long long>(gk) * lda] : 0.0;
    }
#pragma unroll
    for (int r = 0; r < (TN * TK) / (TX * TY); ++r) {   // B tile, coalesced along k
      const int e = tid + r * TX * TY, k = e % TK, n = e / TK;
      const int gk = k0 + k, gn = n0 + n;
      Bs[k][n] = (gk < K && gn < N) ? B[gk + static_cast<long long>(gn) * ldb] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      double av[4], bv[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) av[r] = As[kk][tx + TX * r];
#pragma unroll
      for (int c = 0; c < 4; ++c) bv[c] = Bs[kk][ty + TY * c];
#pragma unroll
      for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[r][c] = fma(av[r], bv[c], acc[r][c]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int gn = n0 + ty + TY * c;
    if (gn >= N) continue;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int gm = m0 + tx + TX * r;
      if (gm >= M) continue;
      double* p = C + gm + static_cast<long long>(gn) * ldc;
      *p = accumulate ? *p + acc[r][c] : acc[r][c];
    }
  }
}

// 1 / m in float64 without a division: the float32 reciprocal of the leading 24
// bits as the seed r0 (relative error below 2^-21) and one third-order step
// r0 (1 + e + e^2), e = 1 - m r0, whose error e^3 is below the float64 rounding.
// The seed's conversions are integer operations, so a reciprocal costs the
// float64 pipe three FMAs.  Pivots outside the float32 range take the division.
__device__ __forceinline__ double recip_fp64(double m) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(m));
  const unsigned e = static_cast<unsigned>(b >> 52) & 0x7ffu;
  if (e - 900u > 240u) return 1.0 / m;
  const float fm = __uint_as_float((static_cast<unsigned>(b >> 63) << 31) | ((e - 896u) << 23) |
                                   (static_cast<unsigned>(b >> 29) & 0x7fffffu));
  const double r0 = f2d_int(__fdividef(1.0f, fm));
  const double d = fma(-m, r0, 1.0);
  return fma(r0, fma(d, d, d), r0);
}

// One thread per (i, j) line, or with SPLIT two (threadIdx.y), which eliminate from
// its two ends and meet in the middle: the upper one rows 0 .. h-1 downwards, the lower one rows
// nz-1 .. h upwards; the two rows that meet are solved as a 2 x 2 system and each
// half is then substituted back outwards.  Elimination
// keeps the reciprocal pivots in `inv` and d' in `out`; back substitution
// overwrites `out`.  With KEPT the reciprocal pivots are already in `inv` (from
// an earlier call with the same coefficients and sizes) and are only read.  The
// singular line (null_i, null_j) is first projected to compatible form (its
// dz-weighted mean removed, recorded in *defect), the unknown where its
// elimination breaks down (the last, or row h) is set to zero, and the result is
// shifted to zero dz-weighted mean.  The beta-scaled z rows are staged in shared memory once per
// block (3 Nz doubles, dynamic) when ROWS is set.  f may alias out (each element
// is read before the same thread writes it).
//
// GB300's float64 pipe (2 FMA a cycle per SM) bounds large fields: 11 operations
// a point, 5 with KEPT, where the loads (24 B a point) come near the pipe.
// Small ones are bound by the chain along a line, which SPLIT halves; rows are
// also read kAhead at a time, one group ahead of the sweep (the loads
// of a row waited for the row before: 2300 cycles a row), and the blocks are
// small enough to reach every SM.  512^3 3.53 -> 2.73
// ms, 1.31 with KEPT; 61x97x75 83 -> 27 and 20 us (SPLIT).
constexpr int kAhead = 8;
constexpr size_t kRowsSmem = 48 * 1024;   // largest z rows staged in shared memory (2048 points)
template <bool ROWS, bool KEPT, bool SPLIT>
__global__ void __launch_bounds__(128)
thomas_fp64_kernel(int nx, int ny, int nz, const double* f, double* out,
                   double* inv, const double* __restrict__ lamx,
                   const double* __restrict__ lamy, const double* __restrict__ az,
                   const double* __restrict__ bz, const double* __restrict__ cz,
                   const double* __restrict__ dz, double alpha, double beta, int null_i,
                   int null_j, double null_scale, double* defect) {
  extern __shared__ double zrow[];   // beta a, beta b, beta c (ROWS; plan tables)
  __shared__ double meet[2][2][SPLIT ? 64 : 1];   // c' and d' of the rows that meet
  if (ROWS) {
    const int tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    for (int k = tid; k < nz; k += nt) {
      zrow[k] = k > 0 ? beta * az[k] : 0.0;
      zrow[nz + k] = beta * bz[k];
      zrow[2 * nz + k] = k < nz - 1 ? beta * cz[k] : 0.0;
    }
    __syncthreads();
  }
  const bool lower = SPLIT && threadIdx.y == 1;
  const int h = SPLIT ? (nz + 1) / 2 : nz;
  const int rows = lower ? nz - h : h;               // of this thread
  const int first = lower ? nz - 1 : 0, dir = lower ? -1 : 1;
  // coupling to the row before (in the sweep's direction), diagonal, and to the next
  auto ra = [&](int k) { return ROWS ? zrow[k] : (k > 0 ? beta * az[k] : 0.0); };
  auto rb = [&](int k) { return ROWS ? zrow[nz + k] : beta * bz[k]; };
  auto rc = [&](int k) { return ROWS ? zrow[2 * nz + k] : (k < nz - 1 ? beta * cz[k] : 0.0); };
  auto before = [&](int k) { return lower ? rc(k) : ra(k); };
  auto after = [&](int k) { return lower ? ra(k) : rc(k); };
  const long long lines = static_cast<long long>(nx) * ny;
  const long long line = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  const bool active = line < lines;
  const int i = static_cast<int>(line % nx), j = static_cast<int>(line / nx);
  const bool is_null = active && i == null_i && j == null_j;
  const double shift = active ? alpha + beta * (lamx[i] + lamy[j]) : 1.0;
  double fshift = 0.0;
  if (is_null) {
    double s = 0.0, w = 0.0;
    for (int k = 0; k < nz; ++k) {
      s = fma(dz[k], f[line + k * lines], s);
      w += dz[k];
    }
    fshift = s / w;
    if (defect && !lower) *defect = fshift * null_scale;
  }
  if (SPLIT && null_i >= 0) __syncthreads();         // both threads have read the line before it is overwritten
  const double* fl = f + line;
  double* ol = out + line;
  double* il = inv + line;
  double fv[kAhead], iv[kAhead];       // rows of the coming group
  auto fetch = [&](int t0) {
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const bool ok = active && t0 + u < rows;
      const long long o = static_cast<long long>(first + dir * (t0 + u)) * lines;
      fv[u] = ok ? fl[o] : 0.0;
      if (KEPT) iv[u] = ok ? il[o] : 0.0;
    }
  };
  double cp = 0.0, dp = 0.0;
  fetch(0);
  for (int t0 = 0; t0 < rows; t0 += kAhead) {
    double fc[kAhead], ic[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      fc[u] = fv[u];
      ic[u] = KEPT ? iv[u] : 0.0;
    }
    fetch(t0 + kAhead);
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int k = first + dir * (t0 + u);
      if (active && t0 + u < rows) {
        const double sub = before(k);
        const double fo = is_null ? fc[u] - fshift : fc[u];
        const double rhs = fma(-sub, dp, fo);
        if (!KEPT) {
          ic[u] = recip_fp64(fma(-sub, cp, rb(k) + shift));
          if (!SPLIT && is_null && k == nz - 1) ic[u] = 0.0;   // vanishing final pivot
          il[k * lines] = ic[u];
        }
        if (!KEPT || (SPLIT && t0 + u == rows - 1)) cp = after(k) * ic[u];
        dp = rhs * ic[u];
        ol[k * lines] = dp;
      }
    }
  }
  // x_{h-1} = d' - c' x_h from above, x_h = d'' - c'' x_{h-1} from below
  if (SPLIT) {
    meet[threadIdx.y][0][threadIdx.x] = cp;
    meet[threadIdx.y][1][threadIdx.x] = dp;
    __syncthreads();
  }
  double x = dp;
  if (SPLIT) {
    const double co = meet[1 - threadIdx.y][0][threadIdx.x], dn = meet[1 - threadIdx.y][1][threadIdx.x];
    if (is_null) x = lower ? 0.0 : dp;               // the determinant vanishes: x_h = 0
    else if (active) x = fma(-cp, dn, dp) * recip_fp64(fma(-cp, co, 1.0));
    if (active) ol[(first + dir * (rows - 1)) * lines] = x;
  }
  // back substitution x_k = d'_k - (after_k inv_k) x_next, outwards from the middle
  auto fetch_back = [&](int t0) {
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const bool ok = active && t0 - u >= 0;
      const long long o = static_cast<long long>(first + dir * (t0 - u)) * lines;
      fv[u] = ok ? ol[o] : 0.0;
      iv[u] = ok ? il[o] : 0.0;
    }
  };
  fetch_back(rows - 2);
  for (int t0 = rows - 2; t0 >= 0; t0 -= kAhead) {
    double fc[kAhead], ic[kAhead];
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      fc[u] = fv[u];
      ic[u] = iv[u];
    }
    fetch_back(t0 - kAhead);
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int k = first + dir * (t0 - u);
      if (active && t0 - u >= 0) {
        x = fma(-(after(k) * ic[u]), x, fc[u]);
        ol[k * lines] = x;
      }
    }
  }
  if (null_i >= 0) {
    if (SPLIT) __syncthreads();                      // both halves of the null line are in place
    if (is_null && !lower) {
      double xs = 0.0, w = 0.0;
      for (int k = 0; k < nz; ++k) {
        xs = fma(dz[k], ol[k * lines], xs);
        w += dz[k];
      }
      const double mean = xs / w;
      for (int k = 0; k < nz; ++k) ol[k * lines] -= mean;
    }
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// r = (f - fshift) - (alpha phi + beta (Lx + Ly + Lz) phi); one thread per
// (i, j) marching along kseg planes (blockIdx.z picks them).  End couplings of non-periodic directions are zero,
// so wrapped neighbour indices only ever meet a zero coefficient.  The rows
// of x and y are read once per thread, those of z once per block (shared memory
// when ROWS).  A point costs nine operations for L phi and one to take beta L phi
// off f on GB300's float64 pipe (~1/64 of the float32 rate, the bound of this
// kernel), one more for alpha phi or for the shift of a singular problem, and one
// for sum r^2 where it is read (SUMS).  A refined solution carries this kernel's
// rounding, so the order is the one that leaves the smallest partial sums: each
// direction's second difference complete before the next, its diagonal between its
// neighbours, f last; and beta multiplies the sum, not the rows, whose rounding
// would be the same at every refinement.  Error of a refined solve in the 2-norm,
// 64^3 uniform points Helmholtz / Dirichlet Poisson / 96 x 100 x 40 stretched
// Helmholtz: 1.4e-16 / 2.0e-16 / 2.2e-16; with beta-scaled rows, f first and the
// diagonals last 3.3e-16 / 2.1e-15 / 5.5e-15 (one operation less, two for
// Helmholtz: 256^3 Poisson 3657 us, this 3694); with the neighbours, one summed
// diagonal, then f 2.6e-16 / 5.1e-16 / 4.5e-15.  The loads of a plane are issued
// a plane ahead.  sums[0] += sum r^2; with ALL also sums[1] += sum r and
// sums[2] += sum vol*r.
template <bool ROWS, bool SUMS, bool ALL>
__global__ void __launch_bounds__(128)
residual_fp64_kernel(int nx, int ny, int nz, const double* __restrict__ f,
                     const double* __restrict__ phi, double* __restrict__ r,
                     const double* __restrict__ rx, const double* __restrict__ ry,
                     const double* __restrict__ rz, const double* __restrict__ dxf,
                     const double* __restrict__ dyf, const double* __restrict__ dzf,
                     double alpha, double beta, const double* __restrict__ fshift_p,
                     double* sums, int kseg) {
  extern __shared__ double zrow[];   // a_k, b_k, c_k (ROWS)
  const int k0 = blockIdx.z * kseg, k1 = min(nz, k0 + kseg);
  if (ROWS) {
    const int tid = threadIdx.x + blockDim.x * threadIdx.y, nt = blockDim.x * blockDim.y;
    for (int k = k0 + tid; k < k1; k += nt) {
      zrow[k] = rz[k];
      zrow[nz + k] = rz[nz + k];
      zrow[2 * nz + k] = rz[2 * nz + k];
    }
    __syncthreads();
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  double s2 = 0.0, s1 = 0.0, sv = 0.0;
  if (i < nx && j < ny) {
    const long long sy = nx, sz = static_cast<long long>(nx) * ny;
    const long long base = i + sy * j;
    const int im = (i == 0) ? nx - 1 : i - 1, ip = (i == nx - 1) ? 0 : i + 1;
    const int jm = (j == 0) ? ny - 1 : j - 1, jp = (j == ny - 1) ? 0 : j + 1;
    const double ax = rx[i], bx = rx[nx + i], cx = rx[2 * nx + i];
    const double ay = ry[j], by = ry[ny + j], cy = ry[2 * ny + j];
    const double fshift = fshift_p ? *fshift_p : 0.0;
    const double vxy = ALL ? dxf[i] * dyf[j] : 0.0;
    double pm = phi[base + sz * (k0 == 0 ? nz - 1 : k0 - 1)];   // k = 0: wrap partner, multiplied by a_0 = 0
    double p0 = phi[base + sz * k0];
    // the loads of a plane are issued one plane ahead of their use
    const double* fq = f + base + sz * k0;
    const double* q = phi + sz * k0;
    const long long xm = im + sy * j, xp = ip + sy * j, ym = i + sy * jm, yp = i + sy * jp;
    double fn = *fq, nxm = q[xm], nxp = q[xp], nym = q[ym], nyp = q[yp];
    for (int k = k0; k < k1; ++k) {
      const long long o = base + sz * k;
      const double fk = fn, vxm = nxm, vxp = nxp, vym = nym, vyp = nyp;
      const long long step = k + 1 < k1 ? sz : 0;
      fq += step;
      q += step;
      fn = *fq, nxm = q[xm], nxp = q[xp], nym = q[ym], nyp = q[yp];
      const double pp = phi[base + sz * ((k == nz - 1) ? 0 : k + 1)];
      const double az = ROWS ? zrow[k] : rz[k];
      const double bz = ROWS ? zrow[nz + k] : rz[nz + k];
      const double cz = ROWS ? zrow[2 * nz + k] : rz[2 * nz + k];
      double acc = ax * vxm;
      acc = fma(bx, p0, acc);
      acc = fma(cx, vxp, acc);
      acc = fma(ay, vym, acc);
      acc = fma(by, p0, acc);
      acc = fma(cy, vyp, acc);
      acc = fma(az, pm, acc);
      acc = fma(bz, p0, acc);
      acc = fma(cz, pp, acc);
      const double rest = fshift_p ? fk - fshift : alpha != 0.0 ? fma(-alpha, p0, fk) : fk;
      const double val = fma(-beta, acc, rest);
      r[o] = val;
      if (SUMS) s2 = fma(val, val, s2);
      if (ALL) {
        s1 += val;
        sv = fma(vxy * dzf[k], val, sv);
      }
      pm = p0;
      p0 = pp;
    }
  }
  if (SUMS) {
    s2 = warp_sum(s2);
    if (ALL) {
      s1 = warp_sum(s1);
      sv = warp_sum(sv);
    }
    if ((threadIdx.x + blockDim.x * threadIdx.y) % 32 == 0) {
      atomicAdd(&sums[0], s2);
      if (ALL) {
        atomicAdd(&sums[1], s1);
        atomicAdd(&sums[2], sv);
      }
    }
  }
}

// sums[0] += sum f^2 and, with ALL, sums[1] += sum f, sums[2] += sum vol*f: one
// warp per x-line (its weight dy_j dz_k once a line), one atomic per block and
// sum.  One float64 operation a point, three with ALL; the pipe bounds it.
template <bool ALL>
__global__ void __launch_bounds__(256)
field_sums_kernel(int nx, int ny, long long lines, const double* __restrict__ f, const double* __restrict__ dxf,
                  const double* __restrict__ dyf, const double* __restrict__ dzf, double* sums) {
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  double s2 = 0.0, s1 = 0.0, sv = 0.0;
  for (long long L = blockIdx.x * 8LL + warp; L < lines; L += gridDim.x * 8LL) {
    const double* row = f + L * nx;
    double sl = 0.0;
    for (int i = lane; i < nx; i += 32) {
      const double v = row[i];
      s2 = fma(v, v, s2);
      if (ALL) {
        s1 += v;
        sl = fma(dxf[i], v, sl);
      }
    }
    if (ALL) sv = fma(dyf[L % ny] * dzf[L / ny], sl, sv);
  }
  __shared__ double sh[3][8];
  s2 = warp_sum(s2);
  if (ALL) {
    s1 = warp_sum(s1);
    sv = warp_sum(sv);
  }
  if (lane == 0) {
    sh[0][warp] = s2;
    sh[1][warp] = s1;
    sh[2][warp] = sv;
  }
  __syncthreads();
  if (threadIdx.x < (ALL ? 3 : 1)) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += sh[threadIdx.x][w];
    atomicAdd(&sums[threadIdx.x], t);
  }
}

// Canonical gauge (reading R4): the volume-weighted mean of phi to within 6 u of
// the mean of |phi| (u = 2^-53), whatever the cancellation and the sizes, in two
// deterministic levels.  A lane of the warp that sums an x-line takes its values
// two at a time (two roundings) into a compensated sum (Kahan: 2 u of the sum of
// magnitudes for any order and length); the lines, weighted by dy dz (two
// roundings), meet in error-free additions (TwoSum) as (hi, lo) pairs per block,
// then one block over them.  2.5 operations of the float64 pipe a point, which
// bounds the kernel; TwoSum at every point, to 3 u, took nine (512^3 2.21 ms), a
// plain FMA chain along the line, whose bound grows with Nx / 32, one (0.38; a
// 512^3 solve 33.10 ms, this 33.46).
__device__ __forceinline__ void two_sum_d(double a, double b, double& s, double& e) {
  s = a + b;
  const double bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}
__device__ __forceinline__ void pair_add_d(double& hi, double& lo, double h2, double l2) {
  double s, e;
  two_sum_d(hi, h2, s, e);
  hi = s;
  lo += e + l2;
}

__global__ void __launch_bounds__(256)
wsum_partial_fp64_kernel(int nx, int ny, int nz, const double* __restrict__ phi, const double* __restrict__ dxf,
                         const double* __restrict__ dyf, const double* __restrict__ dzf, double2* partial) {
  const long long lines = static_cast<long long>(ny) * nz;
  const int lane = threadIdx.x % 32;
  double hi = 0.0, lo = 0.0;
  for (long long L = blockIdx.x * 8LL + threadIdx.x / 32; L < lines; L += gridDim.x * 8LL) {   // x-line (j, k)
    const double* row = phi + static_cast<long long>(nx) * L;
    double sl = 0.0, c = 0.0;            // the lane's share is sl - c
#pragma unroll 4
    for (int i = lane; i < nx; i += 64) {
      double y = fma(dxf[i], row[i], -c);
      if (i + 32 < nx) y = fma(dxf[i + 32], row[i + 32], y);
      const double t = sl + y;
      c = (t - sl) - y;
      sl = t;
    }
    const double wyz = dyf[L % ny] * dzf[L / ny];
    double s, e;
    two_sum_d(hi, wyz * sl, s, e);
    hi = s;
    lo += fma(-wyz, c, e);
  }
  __shared__ double sh[2][256];
  sh[0][threadIdx.x] = hi;
  sh[1][threadIdx.x] = lo;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      double h = sh[0][threadIdx.x], l = sh[1][threadIdx.x];
      pair_add_d(h, l, sh[0][threadIdx.x + w], sh[1][threadIdx.x + w]);
      sh[0][threadIdx.x] = h;
      sh[1][threadIdx.x] = l;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) partial[blockIdx.x] = make_double2(sh[0][0], sh[1][0]);
}

// mean = (sum of the partial pairs) / volume, one block
__global__ void __launch_bounds__(256)
wsum_final_fp64_kernel(int nb, const double2* __restrict__ partial, double inv_vol, double* mean) {
  double hi = 0.0, lo = 0.0;
  for (int b = threadIdx.x; b < nb; b += blockDim.x) pair_add_d(hi, lo, partial[b].x, partial[b].y);
  __shared__ double sh[2][256];
  sh[0][threadIdx.x] = hi;
  sh[1][threadIdx.x] = lo;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      double h = sh[0][threadIdx.x], l = sh[1][threadIdx.x];
      pair_add_d(h, l, sh[0][threadIdx.x + w], sh[1][threadIdx.x + w]);
      sh[0][threadIdx.x] = h;
      sh[1][threadIdx.x] = l;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *mean = (sh[0][0] + sh[1][0]) * inv_vol;
}

__global__ void __launch_bounds__(256) sub_scalar_kernel(long long n, const double* __restrict__ c,
                                                          double* __restrict__ x) {
  const double v = *c;
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n; i += stride)
    x[i] -= v;
}

}  // namespace

namespace {
__global__ void __launch_bounds__(256) add_kernel(long long n, const double* __restrict__ in, double* __restrict__ out) {
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  for (long long i = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; i < n; i += stride)
    out[i] += in[i];
}
}  // namespace

cudaError_t add_fp64(long long n, const double* in, double* out, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const long long blocks = (n + 255) / 256;
  note_launch(1);
  add_kernel<<<static_cast<unsigned>(blocks < 4096 ? blocks : 4096), 256, 0, s>>>(n, in, out);
  return cudaGetLastError();
}

cudaError_t remove_weighted_mean(const tpt_plan_s* p, double* phi, void* scratch, size_t scratch_bytes,
                                 double* mean, cudaStream_t s) {
  int dev_sms = 152;
  cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, p->dev);
  const long long lines = static_cast<long long>(p->n[1]) * p->n[2];
  long long cap = static_cast<long long>(scratch_bytes / sizeof(double2));
  if (cap > 4LL * dev_sms) cap = 4LL * dev_sms;
  if (cap < 1) return cudaErrorInvalidValue;
  const int nb = static_cast<int>((lines + 7) / 8 < cap ? (lines + 7) / 8 : cap);
  double2* partial = static_cast<double2*>(scratch);
  note_launch(3);
  wsum_partial_fp64_kernel<<<nb, 256, 0, s>>>(p->n[0], p->n[1], p->n[2], phi, p->d_dxf[0], p->d_dxf[1],
                                              p->d_dxf[2], partial);
  wsum_final_fp64_kernel<<<1, 256, 0, s>>>(nb, partial, 1.0 / p->vol, mean);
  const long long n = static_cast<long long>(p->n[0]) * p->n[1] * p->n[2];
  long long g = (n + 255) / 256;
  if (g > 16LL * dev_sms) g = 16LL * dev_sms;
  sub_scalar_kernel<<<static_cast<unsigned>(g), 256, 0, s>>>(n, mean, phi);
  return cudaGetLastError();
}

cudaError_t field_sums(const tpt_plan_s* p, const double* f, double* sums, cudaStream_t s) {
  int dev_sms = 152;
  cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, p->dev);
  const long long lines = static_cast<long long>(p->n[1]) * p->n[2];
  long long nb = (lines + 7) / 8;
  if (nb > 8LL * dev_sms) nb = 8LL * dev_sms;
  note_launch();
  auto kern = p->singular ? field_sums_kernel<true> : field_sums_kernel<false>;   // only then are the others read
  kern<<<static_cast<unsigned>(nb), 256, 0, s>>>(p->n[0], p->n[1], lines, f, p->d_dxf[0], p->d_dxf[1], p->d_dxf[2],
                                                 sums);
  return cudaGetLastError();
}

cudaError_t dgemm_cm(int M, int N, int K, const double* A, int lda, long long sA,
                     const double* B, int ldb, long long sB, double* C, int ldc, long long sC,
                     int batch, bool accumulate, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0 || batch <= 0) return cudaSuccess;
  if (batch > 65535) return cudaErrorInvalidConfiguration;
  // split N so that the grid's y extent stays within the hardware limit
  const int nchunk = 65535 * TN;
  for (int n0 = 0; n0 < N; n0 += nchunk) {
    const int nn = (N - n0 < nchunk) ? N - n0 : nchunk;
    dim3 grid((M + TM - 1) / TM, (nn + TN - 1) / TN, batch);
    note_launch();
    dgemm_cm_kernel<<<grid, dim3(TX, TY), 0, s>>>(M, nn, K, A, lda, sA,
                                                  B + static_cast<long long>(n0) * ldb, ldb, sB,
                                                  C + static_cast<long long>(n0) * ldc, ldc, sC,
                                                  accumulate ? 1 : 0);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t thomas_fp64(const tpt_plan_s* p, const double* fhat, double* phihat, double* scratch,
                        double* defect, cudaStream_t s, bool kept) {
  const int nx = p->n[0], ny = p->n[1], nz = p->n[2];
  const long long lines = static_cast<long long>(nx) * ny;
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->dev);
  // Two threads a line up to 128 lines per SM, where the chain bounds the kernel
  // (61x97x75 45 -> 27 us and 25 -> 20); above, the float64 pipe does and the extra
  // operations of the meeting cost (a 256^3 Helmholtz solve 3.45 -> 3.54 ms).  Solves
  // of 128 rows, one thread / two: 84 lines per SM 556 / 518 us, 126 739 / 710, 129
  // 852 / 845, 168 1111 / 1102, 263 and 431 the same.
  const bool split = nz > 1 && lines <= 128LL * sms;
  int bs = split ? 64 : 128;
  while (bs > 32 && lines < 2LL * sms * bs) bs /= 2;   // two blocks per SM, down to a warp
  const long long nb = (lines + bs - 1) / bs;
  const double* rz = p->d_rows[2];
  // f-hat of the null line equals (g_x g_y) times the physical constant
  const double null_scale = p->singular ? 1.0 / (p->null_g[0] * p->null_g[1]) : 0.0;
  const size_t rows_bytes = 3 * static_cast<size_t>(nz) * sizeof(double);
  const bool rows = rows_bytes <= kRowsSmem;
  note_launch();
  auto pick = [&](auto r, auto k) {
    return split ? thomas_fp64_kernel<decltype(r)::value, decltype(k)::value, true>
                 : thomas_fp64_kernel<decltype(r)::value, decltype(k)::value, false>;
  };
  auto kern = rows ? (kept ? pick(std::true_type{}, std::true_type{}) : pick(std::true_type{}, std::false_type{}))
                   : (kept ? pick(std::false_type{}, std::true_type{}) : pick(std::false_type{}, std::false_type{}));
  if (rows && split) {
    // without it static and dynamic memory together may take 48 KB, which the
    // 2 KB of `meet` leave short of the rows from 1963 points on
    const cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kRowsSmem));
    if (e != cudaSuccess) return e;
  }
  kern<<<static_cast<unsigned>(nb), dim3(bs, split ? 2 : 1), rows ? rows_bytes : 0, s>>>(
      nx, ny, nz, fhat, phihat, scratch, p->ddir[0].lam, p->ddir[1].lam, rz, rz + nz, rz + 2 * nz,
      p->d_dxf[2], p->alpha, p->beta, p->singular ? p->null_i : -1, p->singular ? p->null_j : -1,
      null_scale, p->singular ? defect : nullptr);
  return cudaGetLastError();
}

cudaError_t residual_fp64(const tpt_plan_s* p, const double* f, const double* phi, double* r,
                          double* sums, const double* fshift, cudaStream_t s, bool all_sums) {
  const int nx = p->n[0], ny = p->n[1], nz = p->n[2];
  dim3 block(32, 4);
  dim3 grid((nx + 31) / 32, (ny + 3) / 4);
  // planes of a block: as many as leave eight blocks per SM (a plane is a
  // dependent chain of loads and float64 operations, ~0.7 us), at least four;
  // 61x97x75 51 -> 15 us, 32^3 27 -> 8.5 us
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, p->dev);
  const long long tiles = static_cast<long long>(grid.x) * grid.y;
  long long segs = (8LL * sms + tiles - 1) / tiles;
  if (segs > (nz + 3) / 4) segs = (nz + 3) / 4;
  const int kseg = static_cast<int>((nz + segs - 1) / segs);
  grid.z = (nz + kseg - 1) / kseg;
  const size_t rows_bytes = 3 * static_cast<size_t>(nz) * sizeof(double);
  const bool rows = rows_bytes <= kRowsSmem;   // within the default dynamic limit: no static memory here
  auto pick = [&](auto ro) {
    constexpr bool R = decltype(ro)::value;
    return !sums ? residual_fp64_kernel<R, false, false>
                 : all_sums ? residual_fp64_kernel<R, true, true> : residual_fp64_kernel<R, true, false>;
  };
  auto kern = rows ? pick(std::true_type{}) : pick(std::false_type{});
  note_launch();
  kern<<<grid, block, rows ? rows_bytes : 0, s>>>(nx, ny, nz, f, phi, r, p->d_rows[0], p->d_rows[1], p->d_rows[2],
                                                 p->d_dxf[0], p->d_dxf[1], p->d_dxf[2], p->alpha, p->beta,
                                                 fshift, sums, kseg);
  return cudaGetLastError();
}

}  // namespace tpt
