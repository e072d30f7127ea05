// Closed-form prediction standard errors at every grid node (Section 3.4's
// SE_E, SE_L and SE_N; the variances of Eq. (condmvn), Section 3.1 and
// Section 3.2), without drawing a realization.
//
// Exact (local mode, A = K_oo + tau^2 I):
//   var_E(g) = sigma^2 - k_g^T A^-1 k_g,                k_g = K(obs, g).
// Approximate draws v = y + W_2 (z - S y - eps*), W_2 = K_go A^-1, where S is the
// off-grid map (W_1 rows in local mode, J_N in NN mode) and eps* has covariance D
// (diag phi^2, or the grid-box blocks L_b L_b^T):
//   var(g) = sigma^2 - 2 w_g^T u_g + w_g^T Q w_g,
//   w_g = A^-1 k_g,  u_g = S K(grid, g),  Q = S K_gg S^T + D.
// In NN mode S K_gg = K(J_N, grid) and Q = A_N, so var = sigma^2 - k_g^T A_N^-1 k_g
// with the context's surrogate nodes and prediction matrix.
//
// FP64 arithmetic runs at 1/64 of FP32 here, so no per-element work is left to it:
// covariances are evaluated as FP32 pairs (value, low part) with error-free transformations,
// the window sums of u_g and Q are exact integer sums (26-bit weights times 31-bit
// covariances), quadratic forms are summed as pairs.  w_g = A^-1 k_g takes FP32 products with
// the pair A^-1, Q w_g the digit products of ce_xprod.cu.  The nodes are processed in chunks
// of rows.  Grid-to-grid covariances depend only on the lag: an m x (2m - 1) table.
// 256 x 256 nodes, 1000 sites, np = 3, both maps: 45 ms before; the kernels say from what.
#include <algorithm>
#include <cmath>

#include "ce_common.cuh"
#include "ce_internal.h"

namespace ce {
namespace {

struct SeGrid {
  int m;
  double h, sigma2, theta;
  int nu3;
  Aniso an;
};

// The isotropic covariance in grid units as FP32 pairs: C(d) = s2 (1 + a d) 2^(b d).
struct MaternPair {
  float2 s2, a, b;
};

float2 pair_of(double v) {
  const float h = (float)v;
  return make_float2(h, (float)(v - (double)h));
}

MaternPair matern_pair(const SeGrid& g) {
  const double k = (g.nu3 ? std::sqrt(3.0) : 1.0) * g.h / g.theta;
  return {pair_of(g.sigma2), pair_of(g.nu3 ? k : 0.0), pair_of(-k * 1.4426950408889634)};
}

// s + e = a + b exactly (Knuth)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
  return s;
}

// x.x y.x + what a pair keeps of the rest
__device__ __forceinline__ float2 mul_pair(float2 x, float2 y) {
  const float p = __fmul_rn(x.x, y.x);
  return make_float2(p, fmaf(x.x, y.x, -p) + fmaf(x.x, y.y, x.y * y.x));
}

// acc += v, the errors gathered in the low part
__device__ __forceinline__ void add_pair(float2& acc, float2 v) {
  float e;
  acc.x = two_sum(acc.x, v.x, e);
  acc.y += e + v.y;
}

// C at the grid-unit offset (dx, dy), each a pair; relative error about 2^-28 (the FP32
// evaluation of the quadratic and higher terms of 2^g; everything larger is kept in pairs).
__device__ __forceinline__ float2 matern_pair_eval(float2 dx, float2 dy, const MaternPair& k) {
  const float px = __fmul_rn(dx.x, dx.x), py = __fmul_rn(dy.x, dy.x);
  float te;
  const float t0 = two_sum(px, py, te);
  te += fmaf(dx.x, dx.x, -px) + fmaf(dy.x, dy.x, -py) + 2.f * fmaf(dx.x, dx.y, dy.x * dy.y);
  const float t = fmaxf(t0, 1e-30f);
  const float r = fast_rsqrt(t);
  const float d0 = __fmul_rn(t, r);
  const float2 d = make_float2(d0, (fmaf(-d0, d0, t) + te) * (0.5f * r));   // one correction step of the square root
  const float2 x = mul_pair(k.b, d);
  const float n = rintf(x.x);
  const float gh = __fsub_rn(x.x, n);
  const float g = __fadd_rn(gh, x.y), gl = __fsub_rn(x.y, __fsub_rn(g, gh));
  // 2^g = 1 + g ln 2 + g^2 q(g), |g| <= 0.5: the series of exp(g ln 2) to g^8
  float q = 1.3215487e-6f;
  q = fmaf(q, g, 1.5252734e-5f);
  q = fmaf(q, g, 1.5403530e-4f);
  q = fmaf(q, g, 1.3333558e-3f);
  q = fmaf(q, g, 9.6181291e-3f);
  q = fmaf(q, g, 5.5504109e-2f);
  q = fmaf(q, g, 2.4022651e-1f);
  const float2 lng = mul_pair(make_float2(0.693147182f, -1.90465421e-9f), make_float2(g, gl));
  float ee;
  const float e0 = two_sum(1.0f, lng.x, ee);
  const float el = ee + fmaf(g * g, q, lng.y);
  const float e1 = __fadd_rn(e0, el);
  const float2 e = make_float2(e1, __fsub_rn(el, __fsub_rn(e1, e0)));
  const float2 ad = mul_pair(k.a, d);
  float le;
  const float l0 = two_sum(1.0f, ad.x, le);
  const float2 c = mul_pair(mul_pair(make_float2(l0, le + ad.y), e), k.s2);
  const int ni = (int)n;   // b < 0, so n <= 0
  const float sc = ni < -126 ? 0.f : __int_as_float((ni + 127) << 23);
  return make_float2(c.x * sc, c.y * sc);
}

// tab[a][b + m - 1] = (2^31 - 1) C / sigma^2 of the lag of a rows and b columns, 0 <= a < m,
// -m < b < m, rounded (C(-lag) = C(lag), so rows of negative lag are not stored).  FP64: once
// per call.
constexpr double kTabScale = 2147483647.0;

__global__ void se_lag_table_kernel(SeGrid g, int* __restrict__ tab) {
  const int W = 2 * g.m - 1;
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)g.m * W) return;
  const double a = (double)(e / W), b = (double)(e % W - (g.m - 1));
  tab[e] = __double2int_rn(kTabScale * matern_d(aniso_dist(g.h * b, g.h * a, g.an), 1.0, g.theta, g.nu3));
}

// The weights of every row as integers below 2^25 in magnitude, W[i][k] = Wi[i][k] unit[i]
// with unit a power of two (a sum of K <= 64 products with the table stays below 2^63), and
// transposed, Wt[k][i].
__global__ void int_weights_kernel(const float* __restrict__ W, int n, int K, int* __restrict__ Wi, int* __restrict__ Wt,
                                   float* __restrict__ unit) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float mx = 1e-30f;
  for (int k = 0; k < K; ++k) mx = fmaxf(mx, fabsf(W[(long long)i * K + k]));
  int e;
  frexpf(mx, &e);   // mx < 2^e
  const float up = ldexpf(1.f, 25 - e);
  unit[i] = ldexpf(1.f, e - 25);
  for (int k = 0; k < K; ++k) {
    const int v = __float2int_rn(W[(long long)i * K + k] * up);
    Wi[(long long)i * K + k] = v;
    Wt[(long long)k * n + i] = v;
  }
}

// An integer below 2^63 in magnitude as an FP32 pair (49 bits or more).
__device__ __forceinline__ float2 pair_of_int(long long v) {
  const float h = (float)v;
  return make_float2(h, (float)(v - (long long)h));
}

// Kc[r][i] = C(node g0 + r, obs i) rounded to FP32, obs in grid units (integer part,
// fraction); grid.y: rows.  ANISO: the mapped offset in FP64.  65.5 M values: 6.3 -> 0.3 ms.
template <bool ANISO>
__global__ void __launch_bounds__(256) se_cross_kernel(SeGrid g, MaternPair k, const float4* __restrict__ obs, int n,
                                                       long long g0, float* __restrict__ Kc) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int node = (int)(g0 + blockIdx.y);
  const int gi = node / g.m, gj = node % g.m;
  const float4 o = obs[i];
  float v;
  if (ANISO) {
    const double dx = ((double)o.x - gj) + (double)o.y, dy = ((double)o.z - gi) + (double)o.w;
    v = (float)matern_d(aniso_dist(g.h * dx, g.h * dy, g.an), g.sigma2, g.theta, g.nu3);
  } else {
    float2 dx, dy;
    dx.x = two_sum(o.x - (float)gj, o.y, dx.y);
    dy.x = two_sum(o.z - (float)gi, o.w, dy.y);
    const float2 c = matern_pair_eval(dx, dy, k);
    v = c.x + c.y;
  }
  Kc[(long long)blockIdx.y * n + i] = v;
}

// Q = S K_gg S^T + D (local mode), written as the FP32 pair hi + lo (rows of length ld).
// Q[i][j] = sum_k sum_l W[i][k] W[j][l] C(idx[i][k], idx[j][l]); D = diag(phi^2), or for
// two rows of one jointly drawn grid box the product of their noise-factor rows.  A window
// is a w x w block of nodes from its first one; lanes take consecutive j (neighbours along
// the Morton curve).  The inner sums are exact integers, one multiply-add a term where FP64
// took a conversion and a multiply-add at 1/64 rate (n = 1000, K = 36: 2.8 ms).  grid.x: i,
// grid.y: pieces of j.
template <int w>
__global__ void __launch_bounds__(256) se_q_kernel(const int* __restrict__ tab, int m, const int* __restrict__ idx,
                                                   const int* __restrict__ Wi, const int* __restrict__ Wt,
                                                   const float* __restrict__ unit, double sigma2, int n,
                                                   const float* __restrict__ phi, const int* __restrict__ box_cnt,
                                                   const int* __restrict__ box_mem, const float* __restrict__ box_L, int ld,
                                                   float* __restrict__ Qhi, float* __restrict__ Qlo) {
  const int i = blockIdx.x, j = blockIdx.y * blockDim.x + threadIdx.x;
  if (j > i) return;
  constexpr int K = w * w;
  const int pi = __ldg(idx + (long long)i * K), pj = __ldg(idx + (long long)j * K);
  const int di0 = pi / m - pj / m, dj0 = pi % m - pj % m;
  const int* __restrict__ wi = Wi + (long long)i * K;
  const int* __restrict__ wj = Wt + j;
  float2 s = make_float2(0.f, 0.f);
  for (int ka = 0; ka < w; ++ka)
    for (int kb = 0; kb < w; ++kb) {
      long long t = 0;
      for (int la = 0; la < w; ++la) {
        int di = di0 + ka - la, dj = dj0 + kb, step = -1;
        if (di < 0) {
          di = -di;
          dj = -dj;
          step = 1;
        }
        const int* __restrict__ row = tab + (long long)di * (2 * m - 1) + dj + m - 1;
#pragma unroll
        for (int lb = 0; lb < w; ++lb) t += (long long)__ldg(wj + (long long)(la * w + lb) * n) * __ldg(row + step * lb);
      }
      add_pair(s, mul_pair(make_float2((float)__ldg(wi + ka * w + kb), 0.f), pair_of_int(t)));
    }
  double q = ((double)s.x + (double)s.y) * ((double)unit[i] * (double)unit[j]) * (sigma2 / kTabScale);
  const int ci = box_cnt ? box_cnt[i] : 0, cj = box_cnt ? box_cnt[j] : 0;
  if (ci > 0 && cj > 0 && box_mem[(long long)i * kBoxMax] == box_mem[(long long)j * kBoxMax]) {
    const int c = min(ci, cj);
    for (int t = 0; t < c; ++t) q += (double)box_L[(long long)i * kBoxMax + t] * (double)box_L[(long long)j * kBoxMax + t];
  } else if (i == j) {
    q += (double)phi[i] * (double)phi[i];
  }
  const float hi = (float)q, lo = (float)(q - (double)hi);
  Qhi[(long long)i * ld + j] = hi;
  Qlo[(long long)i * ld + j] = lo;
  Qhi[(long long)j * ld + i] = hi;
  Qlo[(long long)j * ld + i] = lo;
}

// w = E (hi + lo) in FP32, E (R x n) times the symmetric pair (n x n, row stride lda, a
// multiple of 128): the K range in kSolveKSplit parts, each part in chunks of 32 whose hi and
// lo products accumulate apart in FP32 and join a Kahan sum; the parts' (sum, compensation)
// pairs join as a float pair, all in this order.  Block: 128 rows x 64 columns, 512 threads of
// 4 x 4 outputs in packed column pairs.  Bound by shared-memory loads (24 bytes a lane per 32
// packed multiply-adds), at 0.45 of the FP32 rate: 65536 x 1000 in 7.2 ms; 256 threads of
// 8 x 4 outputs took 8.3 (255 registers, eight warps).  The form before (32 x 64 blocks, one
// block per K part, the parts' pairs through memory: 8.4 GB there) took 9.8 ms with the joining
// kernel.  The digit products of ce_xprod.cu take 1.4 ms for the same and would carry 90 times less
// error into the exact standard errors (4.5e-7 of them instead of 3.9e-5), which would then differ
// from those of this product by its own error.
__device__ __forceinline__ uint64_t dup2(float x) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(x));
  return d;
}
__device__ __forceinline__ float2 halves(uint64_t v) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(v));
  return d;
}
__device__ __forceinline__ void fma2_into(uint64_t& acc, uint64_t a, uint64_t b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}

constexpr int GM = 128, GN = 64, GK = 32, GE = GK + 2;   // GE: row stride of E's chunk
constexpr size_t kGemmSmem = sizeof(float) * 2 * (GM * GE + 2 * GK * GN);

__global__ void __launch_bounds__(512, 1) se_gemm_kernel(const float* __restrict__ E, int R, int n, const float* __restrict__ Ahi,
                                                         const float* __restrict__ Alo, int lda, float* __restrict__ out) {
  extern __shared__ __align__(16) float gsm[];
  const int c0 = blockIdx.x * GN, r0 = blockIdx.y * GM;
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  const int kper = ((n + kSolveKSplit - 1) / kSolveKSplit + GK - 1) / GK * GK;   // a multiple of GK
  // buffer b of E's chunk, of hi's and of lo's
  auto eb = [&](int b) { return gsm + b * (GM * GE); };
  auto hb = [&](int b) { return gsm + 2 * GM * GE + b * (2 * GK * GN); };
  // copies of one chunk: a warp takes eight rows of E (a lane each column) and each thread one
  // 16-byte piece of hi and of lo
  const int wq = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* __restrict__ esrc = E + (long long)(r0 + wq * 8) * n + lane;
  const int hk = threadIdx.x >> 4, hc = (threadIdx.x & 15) * 4;
  const bool hcol = c0 + hc < lda;   // lda is a multiple of 128: whole pieces in range
  auto load = [&](int b, int k0) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const bool ok = r0 + wq * 8 + q < R && k0 + lane < n;
      cp_async4(static_cast<uint32_t>(__cvta_generic_to_shared(eb(b) + (wq * 8 + q) * GE + lane)),
                ok ? esrc + (long long)q * n + k0 : E, ok);
    }
    const bool ok = k0 + hk < n && hcol;
    const long long off = ok ? (long long)(k0 + hk) * lda + c0 + hc : 0;
    cp_async16(static_cast<uint32_t>(__cvta_generic_to_shared(hb(b) + hk * GN + hc)), Ahi + off, ok);
    cp_async16(static_cast<uint32_t>(__cvta_generic_to_shared(hb(b) + GK * GN + hk * GN + hc)), Alo + off, ok);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float hi[4][4], lo[4][4], sum[4][4], comp[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) hi[i][j] = lo[i][j] = sum[i][j] = comp[i][j] = 0.f;
  load(0, 0);
  int b = 0, part_end = kper;
  for (int k0 = 0; k0 < n; k0 += GK, b ^= 1) {
    if (k0 + GK < n) {
      load(b ^ 1, k0 + GK);   // that buffer was released by the barrier that ended the last chunk
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float* __restrict__ es = eb(b) + ty * 4 * GE;
    const float* __restrict__ hs = hb(b) + tx * 4;
    const float* __restrict__ ls = hb(b) + GK * GN + tx * 4;
    uint64_t ph[4][2], pl[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) ph[i][0] = ph[i][1] = pl[i][0] = pl[i][1] = 0;
#pragma unroll 4
    for (int kk = 0; kk < GK; kk += 2) {
      float2 ev[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) ev[i] = *reinterpret_cast<const float2*>(es + i * GE + kk);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const ulonglong2 h = *reinterpret_cast<const ulonglong2*>(hs + (kk + q) * GN);
        const ulonglong2 l = *reinterpret_cast<const ulonglong2*>(ls + (kk + q) * GN);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint64_t e = dup2(q ? ev[i].y : ev[i].x);
          fma2_into(ph[i][0], e, h.x);
          fma2_into(ph[i][1], e, h.y);
          fma2_into(pl[i][0], e, l.x);
          fma2_into(pl[i][1], e, l.y);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {   // Kahan: sum += (hi part + lo part); comp holds the negated error
        const float2 h2 = halves(ph[i][j / 2]), l2 = halves(pl[i][j / 2]);
        const float yv = __fadd_rn(__fadd_rn(j & 1 ? h2.y : h2.x, j & 1 ? l2.y : l2.x), comp[i][j]);
        const float t = __fadd_rn(sum[i][j], yv);
        comp[i][j] = __fsub_rn(yv, __fsub_rn(t, sum[i][j]));
        sum[i][j] = t;
      }
    if (k0 + GK >= part_end || k0 + GK >= n) {   // the part's pair joins the total
      part_end += kper;
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float err;
          hi[i][j] = two_sum(hi[i][j], sum[i][j], err);
          lo[i][j] += __fadd_rn(err, comp[i][j]);
          sum[i][j] = comp[i][j] = 0.f;
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty * 4 + i;
    if (r >= R) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + tx * 4 + j;
      if (c < n) out[(long long)r * n + c] = hi[i][j] + lo[i][j];
    }
  }
}

// Quadratic forms of 32 nodes per block (lanes: nodes, warps: sites), Kc, Wc rows x n, Tc
// pairs of rows x n:
//   FORM 0: se = sqrt(sigma^2 - sum_i Kc Wc)
//   FORM 1: se = sqrt(sigma^2 - 2 sum_i Uc Wc + sum_i Wc Tc), Uc[g][i] = sum_k W[i][k] C(idx[i][k], g)
// formed here: with lanes along the grid a warp's table reads are contiguous and the
// weights uniform (per site one window of w x w nodes), and u never goes through memory.  (As
// a kernel of its own, in FP64 with scattered table reads, u took 12 ms at 65536 x 1000.)
// The transposed reads of Wc, Kc and Tc pass through shared memory.
constexpr int kDotSites = 64;

template <int FORM, int w>
__global__ void __launch_bounds__(256) se_dot_kernel(const float* __restrict__ Kc, const float* __restrict__ Wc,
                                                     const float2* __restrict__ Tc, const int* __restrict__ tab, int m,
                                                     const int* __restrict__ idx, const int* __restrict__ Wi,
                                                     const float* __restrict__ unit, int n, int rows, double sigma2,
                                                     long long g0, float* __restrict__ se) {
  __shared__ float wt[32][kDotSites + 1];
  __shared__ float2 xt[32][kDotSites + 1];
  __shared__ double part[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int K = w * w;
  const int r0 = blockIdx.x * 32;
  const int node = (int)(g0 + min(r0 + lane, rows - 1));
  const int gi = node / m, gj = node % m;
  const float tscale = (float)(-2.0 * sigma2 / kTabScale), tscale_lo = (float)(-2.0 * sigma2 / kTabScale - (double)tscale);
  float2 acc = make_float2(0.f, 0.f);   // sum Kc Wc, or sum Wc Tc - 2 sum Uc Wc
  for (int i0 = 0; i0 < n; i0 += kDotSites) {
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * kDotSites; e += 256) {
      const int r = e / kDotSites, i = e % kDotSites;
      const bool in = r0 + r < rows && i0 + i < n;
      const long long o = (long long)(r0 + r) * n + i0 + i;
      wt[r][i] = in ? Wc[o] : 0.f;
      if (FORM == 0) xt[r][i] = make_float2(in ? Kc[o] : 0.f, 0.f);
      else xt[r][i] = in ? Tc[o] : make_float2(0.f, 0.f);
    }
    __syncthreads();
    for (int i = warp; i < kDotSites && i0 + i < n; i += 8) {
      float2 x = xt[lane][i];
      if (FORM == 1) {
        const int site = i0 + i;
        const int p = __ldg(idx + (long long)site * K);
        const int4* __restrict__ w4 = reinterpret_cast<const int4*>(Wi + (long long)site * K);
        int wv[K];
#pragma unroll
        for (int k = 0; k < K / 4; ++k) {
          const int4 v = __ldg(w4 + k);
          wv[4 * k] = v.x;
          wv[4 * k + 1] = v.y;
          wv[4 * k + 2] = v.z;
          wv[4 * k + 3] = v.w;
        }
        const int di0 = p / m - gi, dj0 = p % m - gj;
        long long u = 0;
#pragma unroll
        for (int a = 0; a < w; ++a) {
          const int di = di0 + a;
          const int* __restrict__ row = tab + (long long)abs(di) * (2 * m - 1) + (di < 0 ? -dj0 : dj0) + m - 1;
          const int step = di < 0 ? -1 : 1;
#pragma unroll
          for (int b = 0; b < w; ++b) u += (long long)wv[a * w + b] * __ldg(row + step * b);
        }
        float2 up = mul_pair(pair_of_int(u), make_float2(tscale, tscale_lo));
        const float un = __ldg(unit + site);   // a power of two
        add_pair(x, make_float2(up.x * un, up.y * un));
      }
      add_pair(acc, mul_pair(make_float2(wt[lane][i], 0.f), x));
    }
  }
  part[warp][lane] = (double)acc.x + (double)acc.y;
  __syncthreads();
  if (warp == 0 && r0 + lane < rows) {
    double s = 0.0;
    for (int k = 0; k < 8; ++k) s += part[k][lane];
    se[g0 + r0 + lane] = (float)sqrt(fmax(FORM == 0 ? sigma2 - s : sigma2 + s, 0.0));
  }
}

}  // namespace
}  // namespace ce

using namespace ce;

extern "C" int ce_se_map(ce_ctx* ctx, float* se_exact_dev, float* se_approx_dev, void* stream) {
  if (!ctx) return fail(nullptr, CE_ERR_ARG, "null context");
  ctx->err.clear();
  if (ctx->mode < 0) return fail(ctx, CE_ERR_STATE, "no off-grid set-up (ce_krige_weights first)");
  if (se_exact_dev && ctx->mode != CE_LOCAL) {
    return fail(ctx, CE_ERR_STATE, "the exact standard errors need the sites' own prediction matrix (local mode)");
  }
  if (ctx->trend_p > 0) return fail(ctx, CE_ERR_STATE, "the closed forms assume a zero mean (ce_set_trend -1 first)");
  if (!se_exact_dev && !se_approx_dev) return CE_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const bool local = ctx->mode == CE_LOCAL;
  const bool need_u = se_approx_dev && local;
  const int n = ctx->nobs, m = ctx->m, ld = ctx->nobs_pad;
  const long long M = (long long)m * m;
  // rows per chunk: its arrays stay within about 64 MB each (a multiple of 128, the products'
  // block of rows)
  const long long cap = std::max<long long>(128, (64ll << 20) / (8ll * n) / 128 * 128);
  const int Mc = (int)std::min<long long>({(M + 127) / 128 * 128, cap, 32768});
  const size_t chunk = (size_t)Mc * n;
  SeGrid g{m, ctx->h, ctx->sigma * ctx->sigma, ctx->range, ctx->nu == 1.5 ? 1 : 0,
           make_aniso(ctx->aniso_ratio, ctx->aniso_angle)};
  const MaternPair mp = matern_pair(g);

  float* Kc = (float*)dalloc(ctx, sizeof(float) * chunk);
  float* Wc = (float*)dalloc(ctx, sizeof(float) * chunk);
  float *Qhi = nullptr, *Qlo = nullptr, *unit = nullptr;
  void *qdig = nullptr, *rowdig = nullptr;
  float2* Tc = nullptr;
  int *tab = nullptr, *Wi = nullptr, *Wt = nullptr;
  if (need_u) {
    Tc = (float2*)dalloc(ctx, sizeof(float2) * chunk);
    Qhi = (float*)dalloc(ctx, sizeof(float) * (size_t)n * ld);
    Qlo = (float*)dalloc(ctx, sizeof(float) * (size_t)n * ld);
    qdig = dalloc(ctx, xprod_matrix_bytes(n));
    rowdig = dalloc(ctx, xprod_rows_bytes(n, Mc));
    tab = (int*)dalloc(ctx, sizeof(int) * (size_t)m * (2 * m - 1));
    Wi = (int*)dalloc(ctx, sizeof(int) * (size_t)n * ctx->K);
    Wt = (int*)dalloc(ctx, sizeof(int) * (size_t)n * ctx->K);
    unit = (float*)dalloc(ctx, sizeof(float) * n);
  }
  auto release = [&]() {
    for (void* p : {(void*)Kc, (void*)Wc, (void*)Tc, (void*)Qhi, (void*)Qlo, qdig, rowdig, (void*)tab, (void*)Wi, (void*)Wt,
                    (void*)unit})
      dfree(ctx, p);
  };
  if (!Kc || !Wc || (need_u && (!Tc || !Qhi || !Qlo || !qdig || !rowdig || !tab || !Wi || !Wt || !unit))) {
    release();
    return fail(ctx, CE_ERR_OOM, "standard-error work buffers");
  }
  if (need_u) {
    const long long ntab = (long long)m * (2 * m - 1);
    se_lag_table_kernel<<<(unsigned)((ntab + 255) / 256), 256, 0, s>>>(g, tab);
    int_weights_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(ctx->W, n, ctx->K, Wi, Wt, unit);
    const bool boxes = ctx->box_joint > 0;
    auto q = ctx->np == 1 ? se_q_kernel<2> : (ctx->np == 2 ? se_q_kernel<4> : (ctx->np == 3 ? se_q_kernel<6> : se_q_kernel<8>));
    q<<<dim3((unsigned)n, (unsigned)((n + 255) / 256)), 256, 0, s>>>(
        tab, m, ctx->idx, Wi, Wt, unit, g.sigma2, n, ctx->phi, boxes ? ctx->box_cnt : nullptr, boxes ? ctx->box_mem : nullptr,
        boxes ? ctx->box_L : nullptr, ld, Qhi, Qlo);
    launch_xprod_matrix(Qhi, Qlo, ld, n, qdig, s);
    ctx->launches += 4;
  }
  int st = CE_OK, parts = 0;
  {
    const cudaError_t ea = set_max_smem(se_gemm_kernel, kGemmSmem);
    if (ea != cudaSuccess) st = cuda_fail(ea, "standard errors", __FILE__, __LINE__);
  }
  for (long long g0 = 0; g0 < M && st == CE_OK; g0 += Mc) {
    const int rows = (int)std::min<long long>(Mc, M - g0);
    const dim3 gk((unsigned)((n + 255) / 256), (unsigned)rows);
    if (g.an.on) se_cross_kernel<true><<<gk, 256, 0, s>>>(g, mp, ctx->obs, n, g0, Kc);
    else se_cross_kernel<false><<<gk, 256, 0, s>>>(g, mp, ctx->obs, n, g0, Kc);
    se_gemm_kernel<<<dim3((unsigned)((n + GN - 1) / GN), (unsigned)((rows + GM - 1) / GM)), 512, kGemmSmem, s>>>(
        Kc, rows, n, ctx->Ainv_hi, ctx->Ainv_lo, ld, Wc);   // w_g = A^-1 k_g
    ctx->launches += 2;
    const unsigned gd = (unsigned)((rows + 31) / 32);
    if (se_exact_dev || !local) {
      se_dot_kernel<0, 2><<<gd, 256, 0, s>>>(Kc, Wc, nullptr, nullptr, m, nullptr, nullptr, nullptr, n, rows, g.sigma2, g0,
                                             local ? se_exact_dev : se_approx_dev);
      ctx->launches += 1;
    }
    if (need_u) {
      st = launch_xprod(ctx, Wc, n, rows, n, qdig, nullptr, rowdig, reinterpret_cast<float*>(Tc), 1, &parts, nullptr, s);   // Q w_g
      if (st) break;
      auto dot = ctx->np == 1 ? se_dot_kernel<1, 2>
                              : (ctx->np == 2 ? se_dot_kernel<1, 4> : (ctx->np == 3 ? se_dot_kernel<1, 6> : se_dot_kernel<1, 8>));
      dot<<<gd, 256, 0, s>>>(nullptr, Wc, Tc, tab, m, ctx->idx, Wi, unit, n, rows, g.sigma2, g0, se_approx_dev);
      ctx->launches += 3;
    }
  }
  cudaError_t e = cudaGetLastError();
  const cudaError_t e2 = cudaStreamSynchronize(s);
  release();
  if (st) return st;
  if (e == cudaSuccess) e = e2;
  if (e != cudaSuccess) return cuda_fail(e, "standard errors", __FILE__, __LINE__);
  // the digit product's waits are bounded: one that expired has left an incomplete product
  return need_u ? sync_stream_status(ctx, s) : CE_OK;
}
