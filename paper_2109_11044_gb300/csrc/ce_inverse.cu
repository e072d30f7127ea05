// FP64 inverse of a symmetric positive definite matrix (the prediction matrix of
// Eq. (condmvn), once per site set) by symmetric block sweeps, with the large products
// on the tensor cores as exact sums of 8-bit digits.
//
// Sweeping the block K of a symmetric matrix M with pivot P = M_KK = C C^T (Cholesky),
// V = M_:K C^-T:
//   M_ij -= V_i V_j^T,  M_iK = V_i C^-1,  M_Kj = (V_j C^-1)^T,  M_KK = -C^-T C^-1   (i, j outside K);
// after every block has been swept M = -A^-1 (Gauss-Jordan elimination on the diagonal;
// the sweep operator of Beaton and Goodnight).  On the rows not yet swept V is the
// Cholesky factor's panel and the update the Cholesky update, whose terms never exceed
// the diagonal.  (With the pivot's explicit inverse, M_ij -= (M_iK P^-1) M_Kj, they grow
// with the pivot's condition: log det was 10 to 200 times less accurate at tau^2 = 1e-6.)
// The scalar pivots are those of the Cholesky factor: they must be positive, and their
// logarithms sum to log det A.  Only the lower triangle is stored.
//
// FP64 arithmetic runs at two multiply-adds per SM and clock on this part, so n^3 flops
// (n = 2000) need 6.4 ms there.  Per block of 64 columns:
//   panel_kernel<0>, <1>  the two 32-column halves of the block swept within its n x 64
//                   panel, FP64: every thread block factors the 32 x 32 pivot itself
//                   (bound by the chain of 32 pivots and by FP64 throughput; a launch of
//                   its own would add its latency), then takes its rows.  The second one
//                   writes the operands of
//   sweep_update_kernel   M -= V V^T for 128 x 64 tiles of the lower triangle: every row
//                   of V is a power of two times an integer of at most 2^55, cut into
//                   seven signed 8-bit digits held exactly in f16.  A digit product
//                   sums 64 terms of at most 2^14, and the at most seven products of one
//                   weight 256^-(t+u) share an FP32 accumulator in tensor memory: below
//                   2^23, so every sum is exact.  The seven accumulators are joined as a
//                   64-bit integer, rounded once to FP64 and subtracted.  Digits past
//                   weight 256^-6 are dropped: the result carries an error of about
//                   2^-54 of the product of the two rows' largest elements, as an FP64
//                   product rounded at every term does.
// What it replaced (right-looking Cholesky of 32-column panels, then two triangular solves
// with the identity, 2.7 times the needed operations, all FP64) took 32 ms at n = 2000.
#include <cuda_fp16.h>

#include <cmath>
#include <vector>

#include "ce_common.cuh"
#include "ce_internal.h"
#include "ce_tc.cuh"

namespace ce {
namespace {

constexpr int kW = 64;        // columns swept per update
constexpr int kH = 32;        // columns swept at a time within the panel
constexpr int kDigits = 7;    // 8-bit digits of an operand
constexpr uint32_t kABlock = 128 * 128, kBBlock = 64 * 128;   // bytes of one digit of a 128-row / 64-row tile
constexpr int kMaxRows = 32;  // panel rows per thread block

// 1 / p for a normal p > 0: the FP32 reciprocal of the mantissa, two Newton steps in FP64.
__device__ __forceinline__ double recip_pos(double p) {
  const long long b = __double_as_longlong(p);
  const double m = __longlong_as_double((b & 0x000fffffffffffffll) | 0x3ff0000000000000ll);   // [1, 2)
  float x0;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x0) : "f"((float)m));
  double x = (double)x0;
  x = fma(x, fma(-m, x, 1.0), x);
  x = fma(x, fma(-m, x, 1.0), x);
  const long long e = 1023 - ((b >> 52) & 0x7ff);   // p = m 2^-e
  return __longlong_as_double(__double_as_longlong(x) + (e << 52));
}

// 1 / sqrt(p) for a normal p > 0, in the same way.
__device__ __forceinline__ double rsqrt_pos(double p) {
  const long long b = __double_as_longlong(p);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;
  const int q = e >> 1;   // p = m 4^q, m in [1, 4)
  const double m = __longlong_as_double((b & 0x000fffffffffffffll) | ((long long)(1023 + (e & 1)) << 52));
  float x0;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(x0) : "f"((float)m));
  double x = (double)x0;
  const double h = 0.5 * m;
  x = fma(x, fma(-h * x, x, 0.5), x);
  x = fma(x, fma(-h * x, x, 0.5), x);
  return __longlong_as_double(__double_as_longlong(x) - ((long long)q << 52));
}

// C^-1 of a 32 x 32 SPD matrix P = C C^T, 256 threads: thread t holds row t / 8, columns
// 4 (t % 8) .. + 3 of P (both triangles) in a[] and returns those of C^-1.  Elimination of
// [P | I] without pivoting, the identity's part kept in the columns already eliminated:
// at pivot k the rows below subtract l_i = a_ik / a_kk times row k.  Row k reaches the
// other rows through shared memory (two buffers: one barrier per pivot); the owner of the
// next pivot forms its reciprocal before the barrier, while other rows still update.
// Warps whose rows are all done skip the arithmetic.  piv (if not null): the 32 pivots.
__device__ __forceinline__ void factor32(double (&a)[4], double (&rowb)[2][kH], double (&rpb)[2], double (&pv)[kH],
                                         double* __restrict__ piv, int* __restrict__ status) {
  const int i = threadIdx.x >> 3, jg = threadIdx.x & 7, lane = threadIdx.x & 31;
  // rolled over groups of four pivots: the code runs once per launch
#pragma unroll 1
  for (int kg = 0; kg < kH / 4; ++kg) {
#pragma unroll
    for (int kr = 0; kr < 4; ++kr) {
      const int k = 4 * kg + kr;
      if (i == k) {
        *reinterpret_cast<double2*>(&rowb[kr & 1][jg * 4]) = make_double2(a[0], a[1]);
        *reinterpret_cast<double2*>(&rowb[kr & 1][jg * 4 + 2]) = make_double2(a[2], a[3]);
        if (jg == kg) {
          double p = a[kr];
          // positive, normal and finite by its bits (an FP64 compare takes 64 cycles of this chain)
          const long long b = __double_as_longlong(p);
          if (b < 0x0010000000000000ll || b >= 0x7ff0000000000000ll) {   // not positive definite
            atomicMax(status, CE_ERR_NOT_SPD);   // an expired wait, which can lead to this, stays the reported one
            p = 1.0;
          }
          rpb[kr & 1] = recip_pos(p);
          pv[k] = p;
          a[kr] = 1.0;
        }
      }
      __syncthreads();
      if ((threadIdx.x >> 5) * 4 + 3 > k) {
        const double2 c01 = *reinterpret_cast<const double2*>(&rowb[kr & 1][jg * 4]);
        const double2 c23 = *reinterpret_cast<const double2*>(&rowb[kr & 1][jg * 4 + 2]);
        const double l = __shfl_sync(0xffffffffu, a[kr], (lane & 24) + kg) * rpb[kr & 1];
        if (i > k) {
          const double c[4] = {c01.x, c01.y, c23.x, c23.y};
#pragma unroll
          for (int j = 0; j < 4; ++j) {   // the next pivot's column first
            const int e = (kr + 1 + j) & 3;
            a[e] = fma(-l, c[e], a[e]);
          }
          if (jg == kg) a[kr] = -l;
        }
      }
    }
  }
  __syncthreads();
  const double p = pv[i];
  const double sc = rsqrt_pos(p);
  if (piv && jg == 0) piv[i] = p;
#pragma unroll
  for (int j = 0; j < 4; ++j) a[j] = jg * 4 + j <= i ? a[j] * sc : 0.0;
}

// Digits of eight values v[0..7] (columns 8 kg ..) of a row whose 64 values are shared by
// eight adjacent lanes: v = x 2^(e - 55), |x| <= 2^55, x = sum_t d_t 256^(6 - t) with
// -128 <= d_t <= 128, d_t as f16 at 16 bytes per digit (dst + t * stride).  Returns e
// (0 for a row of zeros or of values below 2^-400, whose products cannot matter).
__device__ __forceinline__ int store_digits(const double* __restrict__ v, uint8_t* __restrict__ dst, uint32_t stride) {
  int ef = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) ef = max(ef, (int)((__double_as_longlong(v[j]) >> 52) & 0x7ff));
#pragma unroll
  for (int o = 4; o; o >>= 1) ef = max(ef, __shfl_xor_sync(0xffffffffu, ef, o));
  int e = ef - 1022;   // |v| < 2^e
  const bool zero = e < -400;
  if (zero) e = 0;
  uint32_t out[kDigits][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const long long b = __double_as_longlong(v[j]);
    const int f = (int)((b >> 52) & 0x7ff);
    long long x = (b & 0x000fffffffffffffll) | 0x0010000000000000ll;
    const int d = ef - f - 2;   // right shift that leaves 55 bits for the largest exponent
    if (zero || f == 0 || d > 60) x = 0;
    else if (d <= 0) x <<= -d;
    else x = (x + (1ll << (d - 1))) >> d;
    if (b < 0) x = -x;
#pragma unroll
    for (int t = kDigits - 1; t >= 0; --t) {
      const int q = t ? (int)(signed char)(x & 0xff) : (int)x;
      x = (x - q) >> 8;
      const uint32_t h = __half_as_ushort(__int2half_rn(q));
      if (j & 1) out[t][j / 2] |= h << 16;
      else out[t][j / 2] = h;
    }
  }
#pragma unroll
  for (int t = 0; t < kDigits; ++t)
    *reinterpret_cast<uint4*>(dst + (size_t)t * stride) = make_uint4(out[t][0], out[t][1], out[t][2], out[t][3]);
  return e;
}

// 16-byte piece of columns 8 kg .. + 7 of row r in the 128-byte-swizzled K-major layout
__device__ __forceinline__ uint32_t piece(int r, int kg) { return (uint32_t)r * 128u + ((uint32_t)(kg ^ (r & 7)) << 4); }

// Half H of the sweep of columns k0 .. k0 + 63 within their panel (np x 64): H = 0 gathers
// the panel from the lower triangle of M (ld = np) and keeps its half of V in V0 (np x 32);
// H = 1 reads the panel that H = 0 wrote and writes the digits of both halves of V.  rows:
// panel rows per thread block.  FP64-bound: lanes are laid out so that the triangular
// products take equal lengths in every lane of a warp.
template <int H>
__global__ void __launch_bounds__(256) panel_kernel(const double* __restrict__ M, int np, int k0, int rows,
                                                    const double* __restrict__ Pin, double* __restrict__ Pout,
                                                    double* __restrict__ V0, uint8_t* __restrict__ dig, int* __restrict__ dexp,
                                                    double* __restrict__ piv, int* __restrict__ status) {
  __shared__ double rowb[2][kH], rpb[2], pv[kH];
  __shared__ double C[kH][kH + 1], Po[kH][kH + 1], Vt[kH][kH + 1];   // C^-1; the pivot rows' other half; C^-1 Po
  extern __shared__ __align__(16) double rows_smem[];   // rows start 16-byte aligned
  double (*X)[kW + 2] = reinterpret_cast<double (*)[kW + 2]>(rows_smem);
  double (*V)[kW + 2] = X + rows;
  const int t = threadIdx.x;
  const int r0 = blockIdx.x * rows, nr = min(rows, np - r0);
  const int kb = k0 + kH * H;              // first row (and column) of the pivot block
  constexpr int kc = kH * H, oc = kH - kc;  // its columns within the panel, and the others
  double a[4];
  {
    const int i = t >> 3, j0 = (t & 7) * 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (H == 0) {
        const int hi = max(i, j0 + j), lo = min(i, j0 + j);
        a[j] = M[(long long)(kb + hi) * np + kb + lo];
        Po[i][j0 + j] = M[(long long)(k0 + kH + j0 + j) * np + k0 + i];
      } else {
        a[j] = Pin[(long long)(kb + i) * kW + kc + j0 + j];
        Po[i][j0 + j] = Pin[(long long)(kb + i) * kW + oc + j0 + j];
      }
    }
  }
  if (H == 0) {
    if (r0 >= k0 + kW) {   // below the block: rows of M
      for (int e = t; e < nr * kW; e += 256) X[e / kW][e % kW] = M[(long long)(r0 + e / kW) * np + k0 + e % kW];
    } else {               // the transposed element where the row lies above the column
      for (int e = t; e < nr * kW; e += 256) {
        const int c = e / nr, r = e % nr;
        const int gr = r0 + r, gc = k0 + c;
        X[r][c] = M[(long long)max(gr, gc) * np + min(gr, gc)];
      }
    }
  } else {
    for (int e = t; e < nr * kW; e += 256) X[e / kW][e % kW] = Pin[(long long)r0 * kW + e];
    for (int e = t; e < nr * kH; e += 256) V[e / kH][e % kH] = V0[(long long)r0 * kH + e];
  }
  factor32(a, rowb, rpb, pv, blockIdx.x == 0 ? piv + kb : nullptr, status);
  {
    const int i = t >> 3, j0 = (t & 7) * 4;
#pragma unroll
    for (int j = 0; j < 4; ++j) C[i][j0 + j] = a[j];
  }
  __syncthreads();
  // C^-1 Po: warp w the rows w, 15 - w, 16 + w, 31 - w (66 terms a lane in all), lanes the columns
  {
    const int w = t >> 5, c = t & 31;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int l = q == 0 ? w : (q == 1 ? 15 - w : (q == 2 ? 16 + w : 31 - w));
      double v0 = 0.0, v1 = 0.0;
      int m = 0;
      for (; m + 1 <= l; m += 2) {
        v0 = fma(C[l][m], Po[m][c], v0);
        v1 = fma(C[l][m + 1], Po[m + 1][c], v1);
      }
      if (m == l) v0 = fma(C[l][l], Po[l][c], v0);
      Vt[l][c] = v0 + v1;
    }
  }
  // v = x C^-T for a row x outside the pivot block, the column of C^-1 for one inside; a
  // thread takes columns c and 31 - c (33 terms)
  for (int e = t; e < nr * (kH / 2); e += 256) {
    const int r = e / (kH / 2), c = e % (kH / 2), in = r0 + r - kb;
    const int c2 = kH - 1 - c;
    double v = 0.0, w0 = 0.0, w1 = 0.0;
    if (in >= 0 && in < kH) {
      v = C[c][in];
      w0 = C[c2][in];
    } else {
      for (int l = 0; l <= c; ++l) {
        v = fma(X[r][kc + l], C[c][l], v);
        w0 = fma(X[r][kc + l], C[c2][l], w0);
      }
      for (int l = c + 1; l <= c2; ++l) w1 = fma(X[r][kc + l], C[c2][l], w1);
    }
    V[r][kc + c] = v;
    V[r][kc + c2] = w0 + w1;
  }
  __syncthreads();
  for (int e = t; e < nr * (kH / 2); e += 256) {   // the panel's own columns: v C^-1
    const int r = e / (kH / 2), c = e % (kH / 2), in = r0 + r - kb;
    const int c2 = kH - 1 - c;
    double v = 0.0, w = 0.0, u = 0.0;
    for (int l = c; l < c2; ++l) v = fma(V[r][kc + l], C[l][c], v);
    for (int l = c2; l < kH; ++l) {
      u = fma(V[r][kc + l], C[l][c], u);
      w = fma(V[r][kc + l], C[l][c2], w);
    }
    v += u;
    const bool inside = in >= 0 && in < kH;
    X[r][kc + c] = inside ? -v : v;
    X[r][kc + c2] = inside ? -w : w;
  }
  for (int e = t; e < nr * kH; e += 256) {         // the other columns
    const int r = e / kH, c = e % kH, in = r0 + r - kb;
    double y0 = 0.0, y1 = 0.0;
#pragma unroll 8
    for (int l = 0; l < kH; l += 2) {
      y0 = fma(V[r][kc + l], Vt[l][c], y0);
      y1 = fma(V[r][kc + l + 1], Vt[l + 1][c], y1);
    }
    const bool inside = in >= 0 && in < kH;
    X[r][oc + c] = inside ? y0 + y1 : X[r][oc + c] - (y0 + y1);
  }
  __syncthreads();
  for (int e = t; e < nr * kW; e += 256) Pout[(long long)r0 * kW + e] = X[e / kW][e % kW];
  if (H == 0) {
    for (int e = t; e < nr * kH; e += 256) V0[(long long)r0 * kH + e] = V[e / kH][e % kH];
  } else {
    const int r = t >> 3, kg = t & 7;
    // every lane of a warp takes part in the shuffles; rows past nr repeat the last one
    const int rr = min(r, nr - 1), gr = r0 + rr;
    const int e = store_digits(&V[rr][kg * 8], dig + (size_t)(gr >> 6) * kDigits * kBBlock + piece(gr & 63, kg), kBBlock);
    if (kg == 0 && r < nr) dexp[gr] = e;
  }
}

// T 2^e as a double, rounded to nearest; |T| < 2^63, the result normal or zero.
__device__ __forceinline__ double scaled_double(long long T, int e) {
  unsigned long long u = T < 0 ? (unsigned long long)(-T) : (unsigned long long)T;
  const int lz = __clzll((long long)u);
  u <<= (lz & 63);
  const unsigned long long m = (u >> 11) + ((u >> 10) & 1ull);   // 53 bits, the top one implicit
  const unsigned long long bits = ((unsigned long long)(long long)(1023 + 62 - lz + e) << 52) + m;
  return T == 0 ? 0.0 : __longlong_as_double((long long)(bits | ((unsigned long long)T & 0x8000000000000000ull)));
}

// Dynamic shared memory of a panel block: its rows of the panel and of V.
constexpr size_t panel_smem(int rows) { return sizeof(double) * 2 * (size_t)rows * (kW + 2); }

constexpr uint32_t kUpdateSmem = kDigits * (kABlock + kBBlock) + 1024;

// M -= V V^T on the 128 x 64 tile (I, J) of the lower triangle, the swept block's own rows
// and columns taken from the panel P.  Warps 0-7: epilogue, which waits for the products at most
// epi_wait rounds; warp 8: copies and MMA, which has seen both finish (within its own bound)
// before the block frees its tensor memory and exits, also when the epilogue has given up.
__global__ void __launch_bounds__(288) sweep_update_kernel(double* __restrict__ M, int np, int k0, const double* __restrict__ P,
                                                           const uint8_t* __restrict__ dig, const int* __restrict__ dexp,
                                                           uint32_t epi_wait, int* __restrict__ status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  __shared__ __align__(8) uint64_t bars[3];   // A digit 0 and B; A digits 1-6; products done
  __shared__ uint32_t tmem_slot;
  __shared__ int ue[64];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // block b is tile (I, J), J <= 2 I + 1: I (I + 1) tiles precede row I
  int I = (int)((sqrtf(4.f * (float)blockIdx.x + 1.f) - 1.f) * 0.5f);
  while ((long long)I * (I + 1) > (long long)blockIdx.x) --I;
  while ((long long)(I + 1) * (I + 2) <= (long long)blockIdx.x) ++I;
  const int J = (int)((long long)blockIdx.x - (long long)I * (I + 1));
  const int rbase = I * 128, cbase = J * 64;
  if (cbase == k0) {   // the swept columns: straight from the panel
    for (int e = threadIdx.x; e < 128 * 64; e += 288) {
      const int r = rbase + e / 64, c = e % 64;
      if (r >= cbase + c) M[(long long)r * np + cbase + c] = P[(long long)r * kW + c];
    }
    return;
  }
  if (threadIdx.x == 0) {
    for (int b = 0; b < 3; ++b) mbar_init(smem_u32(&bars[b]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (threadIdx.x < 64) ue[threadIdx.x] = dexp[cbase + threadIdx.x];
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  auto wait = [&](int b, uint32_t limit) {
    bool done = false;
    for (uint32_t it = 0; it < limit && !done; ++it) done = mbar_try_for(smem_u32(&bars[b]), 0u, 2000u);
    return done;
  };
  if (warp == 8) {
    if (lane == 0) {
      // the rows' digits: 64-row blocks, two of which make a digit of the 128-row tile
      const uint8_t* va = dig + (size_t)(2 * I) * kDigits * kBBlock;
      const uint32_t sb = base + kDigits * kABlock;
      mbar_arrive_expect_tx(smem_u32(&bars[0]), kDigits * kBBlock + kABlock);
      bulk_g2s(sb, dig + (size_t)J * kDigits * kBBlock, kDigits * kBBlock, smem_u32(&bars[0]));
      mbar_arrive_expect_tx(smem_u32(&bars[1]), (kDigits - 1) * kABlock);
      for (int t = 0; t < kDigits; ++t)
        for (int h = 0; h < 2; ++h)
          bulk_g2s(base + (uint32_t)t * kABlock + (uint32_t)h * kBBlock, va + (size_t)(h * kDigits + t) * kBBlock, kBBlock,
                   smem_u32(&bars[t ? 1 : 0]));
      const uint32_t ibase = (1u << 4) | ((uint32_t)(128 >> 4) << 24);
      bool ok = wait(0, kWaitLimit);
      tc_fence_after();
#pragma unroll 1
      for (int t = 0; t < kDigits; ++t) {
        if (t == 1) {   // waited for in any case: no copy is in flight when the block exits
          ok = wait(1, kWaitLimit) && ok;
          tc_fence_after();
        }
        if (!ok) continue;
        // digit t of the rows times digits 0 .. 6 - t of the columns (adjacent rows of the stage), at most four
        // (256 columns) per product, into accumulators t .. 6
        const int nd = kDigits - t;
#pragma unroll 1
        for (int u = 0; u < nd; u += 4) {
          const int w = min(4, nd - u);
          const uint64_t da = sw128_desc(base + (uint32_t)t * kABlock), db = sw128_desc(sb + (uint32_t)u * kBBlock);
          const uint32_t idesc = ibase | ((uint32_t)(w * 64 >> 3) << 17);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_issue<KIND_F16>(tmem + (uint32_t)(t + u) * 64u, da + 2u * kk, db + 2u * kk, idesc, (t || kk) ? 1u : 0u);
        }
      }
      mma_commit(smem_u32(&bars[2]));
      ok = wait(2, kWaitLimit) && ok;
      if (!ok) atomicMax(status, CE_ERR_TIMEOUT);
    }
    __syncwarp();
  } else {
    const int q = warp & 3, half = warp >> 2;
    const int r = rbase + 32 * q + lane, c0 = cbase + 32 * half;
    double* __restrict__ row = M + (long long)r * np + c0;
    const bool lower = rbase + 32 * q + 31 >= c0;   // the warp's rows reach the lower triangle
    const bool swept_row = r >= k0 && r < k0 + kW;
    // eight columns at a time, the next eight read ahead; not unrolled (the code would not
    // fit the instruction caches, and a block runs it once)
    double2 nxt[4];
    auto read8 = [&](int c) {
#pragma unroll
      for (int g = 0; g < 4; ++g)
        nxt[g] = lower && c0 + c + 2 * g <= r ? *reinterpret_cast<const double2*>(row + c + 2 * g) : make_double2(0.0, 0.0);
    };
    read8(0);
    const int we = dexp[r];
    const bool ok = __all_sync(0xffffffffu, wait(2, epi_wait));
    tc_fence_after();
    if (!ok && lane == 0) atomicMax(status, CE_ERR_TIMEOUT);
    if (ok && lower) {
#pragma unroll 1
      for (int c = 0; c < 32; c += 8) {
        double m[8];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          m[2 * g] = nxt[g].x;
          m[2 * g + 1] = nxt[g].y;
        }
        if (c + 8 < 32) read8(c + 8);
        uint32_t v[kDigits][8];
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
          tmem_ld8(tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(64 * s + 32 * half + c), v[s]);
        tmem_wait_ld();
#pragma unroll
        for (int s = 0; s < kDigits; ++s)
#pragma unroll
          for (int j = 0; j < 8; ++j) asm volatile("" : "+r"(v[s][j]));   // not read before the wait
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          int f[kDigits];
#pragma unroll
          for (int s = 0; s < kDigits; ++s) f[s] = __float2int_rn(__uint_as_float(v[s][j]));
          const int i0 = f[0] * 256 + f[1], i1 = f[2] * 256 + f[3], i2 = f[4] * 256 + f[5];
          const long long T = ((long long)i0 << 32) + ((long long)i1 << 16) + (long long)i2 + (long long)((f[6] + 128) >> 8);
          m[j] -= scaled_double(T, we + ue[32 * half + c + j] - 54);
        }
        if (swept_row) {   // M_Kj, the transpose of the panel's row j
#pragma unroll
          for (int j = 0; j < 8; ++j) m[j] = P[(long long)(c0 + c + j) * kW + (r - k0)];
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (c0 + c + 2 * g + 1 <= r) *reinterpret_cast<double2*>(row + c + 2 * g) = make_double2(m[2 * g], m[2 * g + 1]);
          else if (c0 + c + 2 * g <= r) row[c + 2 * g] = m[2 * g];
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 8) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// The lower triangle of M = -A^-1 (n x n of an np x np array) as the symmetric FP32 pair
// hi + lo (row stride ld), or mirrored and negated in place (hi null).
__global__ void __launch_bounds__(256) finish_inverse_kernel(double* __restrict__ M, int np, int n, float* __restrict__ hi,
                                                             float* __restrict__ lo, int ld) {
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double tile[32][33];
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int y = ty; y < 32; y += 8) {
    const int i = i0 + y, j = j0 + tx;
    tile[y][tx] = (i < n && j < n && j <= i) ? -M[(long long)i * np + j] : 0.0;
  }
  __syncthreads();
  const bool diag = i0 == j0;
  for (int y = ty; y < 32; y += 8) {
    int i = i0 + y, j = j0 + tx;   // the tile itself
    const double v = diag && tx > y ? tile[tx][y] : tile[y][tx];
    if (i < n && j < n) {
      if (hi) {
        const float h = (float)v;
        hi[(long long)i * ld + j] = h;
        lo[(long long)i * ld + j] = (float)(v - (double)h);
      } else {
        M[(long long)i * np + j] = v;
      }
    }
    i = j0 + y;                    // its mirror image
    j = i0 + tx;
    if (!diag && i < n && j < n) {
      const double w = tile[tx][y];
      if (hi) {
        const float h = (float)w;
        hi[(long long)i * ld + j] = h;
        lo[(long long)i * ld + j] = (float)(w - (double)h);
      } else {
        M[(long long)i * np + j] = w;
      }
    }
  }
}

}  // namespace

int spd_inverse_f64(ce_ctx* ctx, double* M, int n, cudaStream_t s, double* logdet) {
  const int np = (n + 127) / 128 * 128;
  CE_CUDA_TRY(cudaMemsetAsync(ctx->setup_status, 0, sizeof(int), s));
  // one block of work memory: two panels, half of V, the digits of V, the pivots, the exponents
  const size_t panel = sizeof(double) * (size_t)np * kW;
  const size_t dig = (size_t)np * kDigits * 128;   // 128 bytes per row and digit
  uint8_t* buf = (uint8_t*)dalloc(ctx, 2 * panel + panel / 2 + dig + (sizeof(double) + sizeof(int)) * (size_t)np);
  if (!buf) return fail(ctx, CE_ERR_OOM, "inverse workspace");
  double* Pa = reinterpret_cast<double*>(buf);
  double* Pb = Pa + (size_t)np * kW;
  double* V0 = Pb + (size_t)np * kW;
  uint8_t* vd = buf + 2 * panel + panel / 2;
  double* piv = reinterpret_cast<double*>(vd + dig);
  int* ve = reinterpret_cast<int*>(piv + np);
  int nsm = 0, dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = set_max_smem(sweep_update_kernel, kUpdateSmem);
  // panel rows per thread block: one block per SM until a block would hold more than kMaxRows
  // (the FP64 units of every SM take part; each block also factors the pivot)
  int rows = nsm > 0 ? (np + nsm - 1) / nsm : kMaxRows;
  rows = rows < 4 ? 4 : (rows > kMaxRows ? kMaxRows : rows);
  const unsigned gp = (unsigned)((np + rows - 1) / rows);
  const unsigned T = (unsigned)(np / 128);
  const size_t shp = panel_smem(rows);
  for (auto k : {panel_kernel<0>, panel_kernel<1>})
    if (e == cudaSuccess) e = set_max_smem(k, panel_smem(kMaxRows));
  for (int k0 = 0; e == cudaSuccess && k0 < n; k0 += kW) {
    panel_kernel<0><<<gp, 256, shp, s>>>(M, np, k0, rows, nullptr, Pa, V0, nullptr, nullptr, piv, ctx->setup_status);
    panel_kernel<1><<<gp, 256, shp, s>>>(M, np, k0, rows, Pa, Pb, V0, vd, ve, piv, ctx->setup_status);
    sweep_update_kernel<<<T * (T + 1), 288, kUpdateSmem, s>>>(M, np, k0, Pb, vd, ve, ctx->wait_limit, ctx->setup_status);
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  int st = 0;
  std::vector<double> hp(n);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&st, ctx->setup_status, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hp.data(), piv, sizeof(double) * n, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  dfree(ctx, buf);
  if (e != cudaSuccess) return cuda_fail(e, "inverse", __FILE__, __LINE__);
  if (st == CE_ERR_NOT_SPD) return fail(ctx, CE_ERR_NOT_SPD, "prediction matrix is not positive definite");
  if (st) return fail(ctx, st, "the inverse reported a device error");
  double ld = 0.0;
  for (int i = 0; i < n; ++i) ld += std::log(hp[i]);
  *logdet = ld;
  return CE_OK;
}

void launch_finish_inverse(double* M, int n, float* hi, float* lo, int ld, cudaStream_t s) {
  const int np = (n + 127) / 128 * 128;
  const unsigned t = (unsigned)((n + 31) / 32);
  finish_inverse_kernel<<<dim3(t, t), 256, 0, s>>>(M, np, n, hi, lo, ld);
}

}  // namespace ce
