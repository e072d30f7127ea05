// Kriging correction, step 5 of Section 2: v_r = y_r + K_go B[:, r] on every
// grid node, with B = A^-1 (z - z*) the weighted residuals (Eq. (condmvn)).
// The grid x site covariance K_go is never stored: each block evaluates the
// Matern covariance (Section 3.3) for its tile of nodes against a chunk of
// sites in shared memory and contracts it with the matching rows of B.
//
// This file holds the plain FP32 form (CUDA cores).  Distances are formed in
// grid units from exact integer node coordinates and the sites' split
// coordinates (integer part + fraction), so each difference is rounded once.
// Each covariance value is evaluated with compensated FP32 arithmetic (below),
// so it carries about one rounding error, not the larger error of the
// hardware approximations: with clustered sites the weights B are large and of
// alternating sign, the sum K_go B cancels by a factor of 10^2-10^3, and every
// random error of a covariance term is amplified by that factor.  Per chunk of
// 32 sites the products accumulate in FP32; chunk sums join the running sum
// with Kahan compensation.
#include <cmath>

#include "ce_common.cuh"
#include "ce_internal.h"

namespace ce {

int launch_correct_tc(ce_ctx* ctx, const float* B, int R, float* y, cudaStream_t s);

namespace {

constexpr int TN64 = 64;   // grid nodes per block of the FP64 form
constexpr int KC = 32;     // sites per chunk

// Matern constants for the compensated evaluation, in grid units:
// C(d) = s2 (1 + a d) 2^(b d), b = b_hi + b_lo held as two floats.
struct MaternFC {
  float s2, a, b_hi, b_lo;
};

// q(g) ~ (2^g - 1) / g on [-0.5005, 0.5005]: a weighted least-squares fit of the
// relative error of 1 + g q(g) against 2^g on Chebyshev nodes, coefficients
// rounded to FP32 (relative error of 1 + g q(g) below 3e-9 in exact arithmetic).
__constant__ float kExp2Q[7] = {0.6931471824645996f,   0.24022650718688965f,    0.055504102259874344f,
                                0.00961803738027811f,  0.0013334081741049886f,  0.00015467044431716204f,
                                1.5165644072112627e-05f};

// Two FP32 values in one 64-bit register pair; each half is rounded as the scalar
// instruction rounds it.
__device__ __forceinline__ uint64_t pack2(float x, float y) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(x), "f"(y));
  return d;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t both(float x) { return pack2(x, x); }
__device__ __forceinline__ uint64_t sub2(uint64_t a, uint64_t b) { return fma2(b, both(-1.f), a); }
// a b - c: two scalar FMAs, whose negated operand is free (the packed one has none)
__device__ __forceinline__ uint64_t fms2(uint64_t a, uint64_t b, uint64_t c) {
  const float2 x = unpack2(a), y = unpack2(b), z = unpack2(c);
  return pack2(fmaf(x.x, y.x, -z.x), fmaf(x.y, y.y, -z.y));
}

// C at the grid-unit offsets (dx, dy) of two nodes.  d^2 is kept as an unevaluated sum
// t + te (error-free products and sum), d = sqrt(t + te) as d0 + d1 (one correction
// step from the hardware reciprocal square root), the exponent b d as x0 + x1
// (error-free product), and 2^(b d) = 2^n 2^g with n = rint(x0) (by the addition of
// 1.5 2^23) and g = (x0 - n) + x1 by the polynomial above.  The result carries about one
// FP32 rounding of relative error.  The packed instructions are explicit, so the compiler
// fuses no product into an FMA (which would break the two-sum identities).
__device__ __forceinline__ uint64_t matern_f_comp2(uint64_t dx, uint64_t dy, const MaternFC& k) {
  const uint64_t px = mul2(dx, dx), ex = fms2(dx, dx, px);
  const uint64_t py = mul2(dy, dy), ey = fms2(dy, dy, py);
  const uint64_t t0 = add2(px, py);
  const uint64_t bp = sub2(t0, px);
  const uint64_t te = add2(add2(sub2(px, sub2(t0, bp)), sub2(py, bp)), add2(ex, ey));
  const float2 tf = unpack2(t0);
  const float ta = fmaxf(tf.x, 1e-30f), tb = fmaxf(tf.y, 1e-30f);
  const uint64_t t = pack2(ta, tb), r = pack2(fast_rsqrt(ta), fast_rsqrt(tb));
  const uint64_t d0 = mul2(t, r);
  const uint64_t d1 = mul2(sub2(te, fms2(d0, d0, t)), mul2(both(0.5f), r));
  const uint64_t bh = both(k.b_hi), a = both(k.a);
  const uint64_t x0 = mul2(bh, d0);
  const uint64_t x1 = add2(fms2(bh, d0, x0), fma2(bh, d1, mul2(both(k.b_lo), d0)));
  const uint64_t mg = add2(x0, both(12582912.f));
  const uint64_t n = add2(mg, both(-12582912.f));
  const uint64_t g = add2(sub2(x0, n), x1);
  uint64_t q = both(kExp2Q[6]);
#pragma unroll
  for (int i = 5; i >= 0; --i) q = fma2(q, g, both(kExp2Q[i]));
  const uint64_t e = fma2(g, q, both(1.0f));
  const uint64_t lin = fma2(a, d0, fma2(a, d1, both(1.0f)));
  // 2^n from the low bits of the shifted sum; b < 0, so n <= 0
  const float2 nf = unpack2(n), mf = unpack2(mg);
  const uint64_t sc = pack2(__int_as_float((__float_as_int(mf.x) - 0x4B400000 + 127) << 23),
                            __int_as_float((__float_as_int(mf.y) - 0x4B400000 + 127) << 23));
  const float2 v = unpack2(mul2(mul2(mul2(both(k.s2), lin), e), sc));
  return pack2(nf.x < -126.f ? 0.f : v.x, nf.y < -126.f ? 0.f : v.y);
}

__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}

// Block: TN nodes x RTILE realizations, threads of TN / 16 nodes x RPT realizations.  Sites go
// in chunks of 32: the covariance tile of the next chunk is evaluated (two nodes at a time in
// packed arithmetic) into one of two buffers while the current one is multiplied, half of the
// warps in one order and half in the other, so that both kinds of work are in flight; the
// weights arrive with cp.async.  Bound by the FP32 pipe (42 operations per covariance, one
// multiply-add per product, four per output and chunk for the Kahan sum) and, in the products,
// by shared-memory loads (64 bytes a lane per 32 packed multiply-adds of an 8 x 8 tile).  Against
// 64-node blocks that evaluated one node at a time and read each weight from its
// realization's row (one transaction per lane): 300 x 300 nodes, 1100 sites, 10 / 50 / 100
// realizations 435 / 876 / 1595 us before, 287 / 680 / 1123 now; 512 x 512, 2000 sites, 128
// realizations 8.77 ms before, 5.26 now; 64 x 64, 200 sites, 10 realizations 31 us before, 22 now.
// The weight of (realization r, site k) is B[r ldr + k ldk].
// Anisotropic covariance (an.x = 1): the grid-unit offset is mapped by the 2 x 2
// matrix (an.y, an.z; an.w, a22) before the evaluation.
template <int RTILE, int RPT>
struct SimtShape {
  static constexpr int NTHREADS = 16 * RTILE / RPT;   // 16 groups of nodes
  static constexpr int MINBLOCKS = RPT == 2 ? 5 : (RPT == 4 ? 4 : (NTHREADS == 256 ? 1 : 2));
};

template <int TN, int RTILE, int RPT>
__global__ void __launch_bounds__(SimtShape<RTILE, RPT>::NTHREADS, SimtShape<RTILE, RPT>::MINBLOCKS)
correct_simt(float* __restrict__ y, int m, const float4* __restrict__ obs, int nobs, const float* __restrict__ B, int ldr, int ldk,
             int R, MaternFC mf, float4 an, float a22) {
  constexpr int NT = SimtShape<RTILE, RPT>::NTHREADS;
  constexpr int TR = RTILE / RPT;                     // threads along the realizations
  constexpr int NP = TN / 32;                         // node pairs per thread
  extern __shared__ __align__(16) float csm[];
  float* const Cs = csm;                              // [2][KC][TN]
  float* const Bs = csm + 2 * KC * TN;                // [2][KC][RTILE]
  const long long M = (long long)m * m;
  const long long g0 = (long long)blockIdx.x * TN;
  const int r0 = blockIdx.y * RTILE;
  const int tn = threadIdx.x % 16, tr = threadIdx.x / 16;
  uint64_t sum[NP][RPT], comp[NP][RPT];   // node pairs x realizations
#pragma unroll
  for (int i = 0; i < NP; ++i)
#pragma unroll
    for (int j = 0; j < RPT; ++j) sum[i][j] = comp[i][j] = 0;
  // every element this thread evaluates belongs to the same two nodes (NT is a multiple of TN / 2)
  const int ep = threadIdx.x % (TN / 2);
  const long long ga = g0 + 2 * ep, gb = ga + 1;
  const uint64_t gi2 = pack2(ga < M ? (float)(int)(ga / m) : 0.f, gb < M ? (float)(int)(gb / m) : 0.f);
  const uint64_t gj2 = pack2(ga < M ? (float)(int)(ga % m) : 0.f, gb < M ? (float)(int)(gb % m) : 0.f);
  auto load_b = [&](int bf, int k0) {
    for (int e = threadIdx.x; e < KC * RTILE; e += NT) {
      const int kk = e / RTILE, rr = e % RTILE;
      const bool ok = k0 + kk < nobs && r0 + rr < R;
      cp_async4(static_cast<uint32_t>(__cvta_generic_to_shared(Bs + (bf * KC + kk) * RTILE + rr)),
                ok ? B + (long long)(r0 + rr) * ldr + (long long)(k0 + kk) * ldk : B, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto evaluate = [&](int bf, int k0) {
#pragma unroll 2
    for (int kk = threadIdx.x / (TN / 2); kk < KC; kk += NT / (TN / 2)) {
      uint64_t c = 0;
      if (k0 + kk < nobs) {
        const float4 o = __ldg(obs + k0 + kk);
        const uint64_t dx = add2(add2(gj2, both(-o.x)), both(-o.y)), dy = add2(add2(gi2, both(-o.z)), both(-o.w));
        c = an.x != 0.f ? matern_f_comp2(fma2(both(an.y), dx, mul2(both(an.z), dy)), fma2(both(an.w), dx, mul2(both(a22), dy)), mf)
                        : matern_f_comp2(dx, dy, mf);
      }
      *reinterpret_cast<uint64_t*>(Cs + (bf * KC + kk) * TN + 2 * ep) = c;
    }
  };
  auto multiply = [&](int bf) {
    uint64_t part[NP][RPT];
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
      for (int j = 0; j < RPT; ++j) part[i][j] = 0;
#pragma unroll 2
    for (int kk = 0; kk < KC; ++kk) {
      // TN = 128: nodes 4 tn .. + 3 and 64 + 4 tn .. + 3; 64: 4 tn .. + 3; 32: 2 tn, 2 tn + 1
      const float* __restrict__ cr = Cs + (bf * KC + kk) * TN;
      uint64_t c[NP];
      if constexpr (NP == 1) {
        c[0] = *reinterpret_cast<const uint64_t*>(cr + 2 * tn);
      } else {
#pragma unroll
        for (int h = 0; h < NP / 2; ++h) {
          const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(cr + 64 * h + 4 * tn);
          c[2 * h] = x.x;
          c[2 * h + 1] = x.y;
        }
      }
      // realizations 4 tr .. + 3 (and RTILE / 2 on), or RPT tr ..
      const float* __restrict__ br = Bs + (bf * KC + kk) * RTILE;
      float b[RPT];
      if constexpr (RPT == 2) {
        const float2 b0 = *reinterpret_cast<const float2*>(br + 2 * tr);
        b[0] = b0.x; b[1] = b0.y;
      } else {
#pragma unroll
        for (int h = 0; h < RPT / 4; ++h) {
          const float4 b0 = *reinterpret_cast<const float4*>(br + h * 4 * TR + 4 * tr);
          b[4 * h] = b0.x; b[4 * h + 1] = b0.y; b[4 * h + 2] = b0.z; b[4 * h + 3] = b0.w;
        }
      }
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        const uint64_t bb = both(b[j]);
#pragma unroll
        for (int i = 0; i < NP; ++i) part[i][j] = fma2(c[i], bb, part[i][j]);
      }
    }
#pragma unroll
    for (int i = 0; i < NP; ++i)
#pragma unroll
      for (int j = 0; j < RPT; ++j) {   // Kahan
        const uint64_t yv = sub2(part[i][j], comp[i][j]);
        const uint64_t t = add2(sum[i][j], yv);
        comp[i][j] = sub2(sub2(t, sum[i][j]), yv);
        sum[i][j] = t;
      }
  };
  load_b(0, 0);
  evaluate(0, 0);
  int bf = 0;
  const int order = (threadIdx.x >> 5) & 1;
  for (int k0 = 0; k0 < nobs; k0 += KC, bf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();   // this chunk's tile and weights are there; the other buffers are free
    const bool more = k0 + KC < nobs;
    if (more) load_b(bf ^ 1, k0 + KC);
#pragma unroll 1
    for (int ph = 0; ph < 2; ++ph) {
      if (ph == order) multiply(bf);
      else if (more) evaluate(bf ^ 1, k0 + KC);
    }
  }
  // per realization all loads in flight before any store
  constexpr int NN = TN / 16;
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int r = r0 + (RPT == 8 ? (j / 4) * 4 * TR + 4 * tr + j % 4 : RPT * tr + j);
    if (r >= R) continue;
    const int n0 = NN == 2 ? 2 * tn : 4 * tn;
    float* __restrict__ yr = y + (long long)r * M + g0 + n0;
    float yv[NN];
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      const int o = (i / 4) * 64 + i % 4;
      yv[i] = g0 + n0 + o < M ? yr[o] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < NN; ++i) {
      const int o = (i / 4) * 64 + i % 4;
      const float2 s2 = unpack2(sum[i / 2][j]);
      if (g0 + n0 + o < M) yr[o] = yv[i] + (i & 1 ? s2.y : s2.x);
    }
  }
}

// Bt[k][r] = B[r][k], k < n, r < R: the order in which the blocks read the weights (rows of R).
__global__ void transpose_b_kernel(const float* __restrict__ B, int ldb, int R, int n, float* __restrict__ Bt) {
  __shared__ float tile[32][33];
  const int k0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  for (int y = threadIdx.y; y < 32; y += 8)
    if (r0 + y < R && k0 + threadIdx.x < n) tile[y][threadIdx.x] = B[(long long)(r0 + y) * ldb + k0 + threadIdx.x];
  __syncthreads();
  for (int y = threadIdx.y; y < 32; y += 8)
    if (k0 + y < n && r0 + threadIdx.x < R) Bt[(long long)(k0 + y) * R + r0 + threadIdx.x] = tile[threadIdx.x][y];
}

// The FP64 form: the same tiling with every step in FP64 (site coordinates from the
// FP64 copy where local Kriging keeps one, the covariance by the closed form of
// Section 3.3 with the library exp, products and sums in FP64), the field read and
// written once in FP32.  RT64 x 16 realizations per block; a comparison form for the
// reduced-precision ones, not a fast path (FP64 runs far below FP32 on this part).
// kh = h sqrt(3) / theta (nu = 3/2) or h / theta (nu = 1/2): C = s2 (1 + t) e^-t or
// s2 e^-t with t = kh times the grid-unit distance.
template <int RT64>
__global__ void __launch_bounds__(256) correct_f64(float* __restrict__ y, int m, const double* __restrict__ sxy,
                                                   const float4* __restrict__ obs, double x0, double y0, double inv_h,
                                                   int nobs, const float* __restrict__ B, int ldb, int R, double sigma2,
                                                   double kh, int nu3, Aniso ad) {
  constexpr int RTILE = 16 * RT64;
  __shared__ double Cs[KC][TN64];
  __shared__ double Bs[KC][RTILE];
  const long long M = (long long)m * m;
  const long long g0 = (long long)blockIdx.x * TN64;
  const int r0 = blockIdx.y * RTILE;
  const int tn = threadIdx.x % 16, tr = threadIdx.x / 16;
  double acc[4][RT64];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < RT64; ++j) acc[i][j] = 0.0;
  const long long gt = g0 + threadIdx.x % TN64;
  const double gti = gt < M ? (double)(gt / m) : 0.0, gtj = gt < M ? (double)(gt % m) : 0.0;
  for (int k0 = 0; k0 < nobs; k0 += KC) {
#pragma unroll
    for (int t = 0; t < KC * TN64 / 256; ++t) {
      const int e = threadIdx.x + 256 * t;
      const int kk = e / TN64, nn = e % TN64;
      double c = 0.0;
      const int q = k0 + kk;
      if (q < nobs && gt < M) {
        double gx, gy;   // the site in grid units
        if (sxy) {
          gx = (sxy[2 * q] - x0) * inv_h;
          gy = (sxy[2 * q + 1] - y0) * inv_h;
        } else {
          const float4 o = obs[q];
          gx = (double)o.x + (double)o.y;
          gy = (double)o.z + (double)o.w;
        }
        const double t = kh * aniso_dist(gtj - gx, gti - gy, ad);
        c = nu3 ? sigma2 * (1.0 + t) * exp(-t) : sigma2 * exp(-t);
      }
      Cs[kk][nn] = c;
    }
    for (int e = threadIdx.x; e < KC * RTILE; e += 256) {
      const int kk = e / RTILE, rr = e % RTILE;
      Bs[kk][rr] = (k0 + kk < nobs && r0 + rr < R) ? (double)B[(long long)(r0 + rr) * ldb + k0 + kk] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < KC; ++kk) {
      double c[4], b[RT64];
#pragma unroll
      for (int i = 0; i < 4; ++i) c[i] = Cs[kk][tn + 16 * i];
#pragma unroll
      for (int j = 0; j < RT64; ++j) b[j] = Bs[kk][tr + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < RT64; ++j) acc[i][j] = fma(c[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < RT64; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = r0 + tr + 16 * j;
      const long long g = g0 + tn + 16 * i;
      if (r < R && g < M) y[(long long)r * M + g] = (float)((double)y[(long long)r * M + g] + acc[i][j]);
    }
}

}  // namespace

MaternF matern_grid_units(const ce_ctx* ctx) {
  MaternF k;
  const double log2e = 1.4426950408889634;
  k.s2 = (float)(ctx->sigma * ctx->sigma);
  if (ctx->nu == 1.5) {
    const double a = std::sqrt(3.0) * ctx->h / ctx->range;
    k.a = (float)a;
    k.b = (float)(-a * log2e);
  } else {
    k.a = 0.f;
    k.b = (float)(-ctx->h / ctx->range * log2e);
  }
  return k;
}

int launch_correct(ce_ctx* ctx, const float* B, int R, float* y, cudaStream_t s) {
  if (ctx->mode == CE_NN && ctx->nn_circulant) return launch_correct_circulant(ctx, B, R, y, s);
  if (ctx->prec == CE_PREC_FP64) {
    const long long M = (long long)ctx->m * ctx->m;
    const Aniso ad = make_aniso(ctx->aniso_ratio, ctx->aniso_angle);
    const double kh = (ctx->nu == 1.5 ? std::sqrt(3.0) : 1.0) * ctx->h / ctx->range;
    const double* sxy = ctx->mode == CE_LOCAL ? ctx->sites64 : nullptr;
    const double s2 = ctx->sigma * ctx->sigma;
    const int nu3 = ctx->nu == 1.5 ? 1 : 0;
    const unsigned gx = (unsigned)((M + TN64 - 1) / TN64);
    if (R <= 16)
      correct_f64<1><<<dim3(gx, 1), 256, 0, s>>>(y, ctx->m, sxy, ctx->obs, ctx->x0, ctx->y0, 1.0 / ctx->h, ctx->nobs, B,
                                                 ctx->nobs_pad, R, s2, kh, nu3, ad);
    else if (R <= 32)
      correct_f64<2><<<dim3(gx, 1), 256, 0, s>>>(y, ctx->m, sxy, ctx->obs, ctx->x0, ctx->y0, 1.0 / ctx->h, ctx->nobs, B,
                                                 ctx->nobs_pad, R, s2, kh, nu3, ad);
    else
      correct_f64<4><<<dim3(gx, (unsigned)((R + 63) / 64)), 256, 0, s>>>(y, ctx->m, sxy, ctx->obs, ctx->x0, ctx->y0,
                                                                         1.0 / ctx->h, ctx->nobs, B, ctx->nobs_pad, R, s2,
                                                                         kh, nu3, ad);
    CE_CUDA_TRY(cudaGetLastError());
    return CE_OK;
  }
  if (ctx->prec != CE_PREC_FP32) return launch_correct_tc(ctx, B, R, y, s);
  const MaternF m1 = matern_grid_units(ctx);
  const double log2e = 1.4426950408889634;
  const double b = (ctx->nu == 1.5 ? -std::sqrt(3.0) : -1.0) * ctx->h / ctx->range * log2e;
  MaternFC mf;
  mf.s2 = m1.s2;
  mf.a = m1.a;
  mf.b_hi = (float)b;
  mf.b_lo = (float)(b - (double)mf.b_hi);
  const long long M = (long long)ctx->m * ctx->m;
  const int ldb = ctx->nobs_pad;
  const Aniso ad = make_aniso(ctx->aniso_ratio, ctx->aniso_angle);
  const float4 an = make_float4(ad.on ? 1.f : 0.f, (float)ad.a11, (float)ad.a12, (float)ad.a21);
  const float a22 = (float)ad.a22;
  // More than 16 realizations: the weights transposed into the residuals' buffer (dead after
  // the solve, R x nobs), so that a chunk's loads are contiguous; a lane per row would touch
  // one line per element.
  const float* Bk = B;
  int ldr = ldb, ldk = 1;
  if (R > 16) {
    transpose_b_kernel<<<dim3((unsigned)((ctx->nobs + 31) / 32), (unsigned)((R + 31) / 32)), dim3(32, 8), 0, s>>>(B, ldb, R, ctx->nobs,
                                                                                                              ctx->E);
    Bk = ctx->E;
    ldr = 1;
    ldk = R;
    ctx->launches += 1;
  }
  int nsm = 0, dev = 0;
  CE_CUDA_TRY(cudaGetDevice(&dev));
  CE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  // The node tile: the widest of its list that still gives every SM two blocks (each output is
  // the same sum in every tile, to the bit).  A tile of 32 nodes is what keeps a small grid
  // busy: 64 x 64 nodes, 200 sites, 10 realizations take 22 us with 32-node blocks and 45 us
  // with 32 blocks of 128.  Up to 16 realizations the evaluation is most of the work and 128
  // nodes halve the loads per value (300 x 300, 1100 sites, 10 realizations: 287 us, 309 with
  // 64); above 64 the 8 x 8 tiles need them (100 realizations: 1123 us, 1375 with 64).  Between,
  // three blocks of 64 nodes per SM are faster than two of 128 (50 realizations: 680 us
  // against 760; 32: 414 against 508).
  auto launch = [&](auto k0, int tn0, auto k1, int tn1, auto k2, int tn2, int rtile, int nthreads) -> int {
    const long long rb = (R + rtile - 1) / rtile;
    auto fills = [&](int tn) { return (M + tn - 1) / tn * rb >= 2 * nsm; };
    const int tn = fills(tn0) ? tn0 : (fills(tn1) ? tn1 : tn2);
    auto kernel = tn == tn0 ? k0 : (tn == tn1 ? k1 : k2);
    const size_t smem = sizeof(float) * 2 * KC * (size_t)(tn + rtile);
    CE_CUDA_TRY(set_max_smem(kernel, smem));
    kernel<<<dim3((unsigned)((M + tn - 1) / tn), (unsigned)rb), nthreads, smem, s>>>(y, ctx->m, ctx->obs, ctx->nobs, Bk, ldr, ldk, R,
                                                                                  mf, an, a22);
    return CE_OK;
  };
  int st;
  if (R <= 16)
    st = launch(correct_simt<128, 16, 2>, 128, correct_simt<64, 16, 2>, 64, correct_simt<32, 16, 2>, 32, 16, SimtShape<16, 2>::NTHREADS);
  else if (R <= 32)
    st = launch(correct_simt<64, 32, 4>, 64, correct_simt<32, 32, 4>, 32, correct_simt<32, 32, 4>, 32, 32, SimtShape<32, 4>::NTHREADS);
  else if (R <= 64)
    st = launch(correct_simt<64, 64, 8>, 64, correct_simt<32, 64, 8>, 32, correct_simt<32, 64, 8>, 32, 64, SimtShape<64, 8>::NTHREADS);
  else
    st = launch(correct_simt<128, 128, 8>, 128, correct_simt<64, 128, 8>, 64, correct_simt<32, 128, 8>, 32, 128,
                SimtShape<128, 8>::NTHREADS);
  if (st) return st;
  ctx->launches += 1;
  CE_CUDA_TRY(cudaGetLastError());
  return CE_OK;
}

}  // namespace ce
