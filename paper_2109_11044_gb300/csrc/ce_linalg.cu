// Dense linear algebra of the Kriging step (Eq. (condmvn); Section 3.1).
//  - FP64, once per site set: the product that maps data to NN surrogate data (the
//    inverse of the prediction matrix itself: ce_inverse.cu).
//  - FP32, per call: B = E (A^-1_hi + A^-1_lo) for the R x n residual block E
//    (A^-1 is symmetric, so this is (A^-1 E^T)^T).  Sums run over 32-term
//    chunks whose partial results are added with Kahan compensation.
#include "ce_common.cuh"
#include "ce_internal.h"
#include "ce_solve_tile.cuh"

namespace ce {
namespace {

// C (M x N, ldc) -= A (M x K, lda) B (K x N, ldb).  64 x 64 tiles, 256 threads, 4 x 4 each.
__global__ void __launch_bounds__(256) gemm64_sub(const double* __restrict__ A, int lda, const double* __restrict__ B, int ldb,
                                                  double* __restrict__ C, int ldc, int M, int N, int K) {
  const int bm = blockIdx.y * 64, bn = blockIdx.x * 64;
  __shared__ double As[16][64 + 1];
  __shared__ double Bs[16][64 + 1];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  double acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += 16) {
    for (int e = threadIdx.x; e < 16 * 64; e += 256) {
      const int kk = e / 64, mm = e % 64;
      const int gm = bm + mm, gk = k0 + kk, gn = bn + mm;
      As[kk][mm] = gm < M && gk < K ? A[(long long)gm * lda + gk] : 0.0;
      Bs[kk][mm] = gn < N && gk < K ? B[(long long)gk * ldb + gn] : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = As[kk][ty + 16 * i]; b[i] = Bs[kk][tx + 16 * i]; }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int gm = bm + ty + 16 * i, gn = bn + tx + 16 * j;
      if (gm < M && gn < N) C[(long long)gm * ldc + gn] -= acc[i][j];
    }
}

template <int CHAIN>
__global__ void __launch_bounds__(128, CHAIN == 4 ? 4 : 5) solve_gemm_f32(const float* __restrict__ E, int R, int n,
                                                      const float* __restrict__ Ahi, const float* __restrict__ Alo,
                                                      int lda, float* __restrict__ part) {
  __shared__ __align__(16) float sm[SV_SMEM / sizeof(float)];
  solve_tile<CHAIN>(E, R, n, Ahi, Alo, lda, part, blockIdx.x * SV_TC, blockIdx.y * SV_TR, blockIdx.z, 0xffffffffu, threadIdx.x, sm,
                    [] { __syncthreads(); });
}

// Bout[r][c] = the partial (sum, compensation) pairs added as an unevaluated
// float pair (TwoSum of the sums, the compensations and the TwoSum errors gathered in
// a second float: FP64 arithmetic is slow on this part), rounded once.  PARTS: their number
// where it is fixed, so that all loads are in flight (1500 rows, R = 60, the whole solve: 45.5 us
// with a runtime count, 43.5 with this one); 0 takes `parts`, or (WIDE) SV_KSPLIT where
// scale[r] < 0.
template <int PARTS, bool WIDE>
__global__ void solve_reduce(const float* __restrict__ part, int parts, const float* __restrict__ scale, int R, int n,
                             float* __restrict__ Bout, int ldb) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long long)R * n) return;
  const int r = (int)(e / n), c = (int)(e % n);
  const long long stride = (long long)R * n;
  const float2* __restrict__ pp = reinterpret_cast<const float2*>(part);
  float hi = 0.f, lo = 0.f;
  auto add = [&](int k) {
    const float2 v = pp[k * stride + e];
    const float t = __fadd_rn(hi, v.x);
    const float z = __fsub_rn(t, hi);
    lo += __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(v.x, z)) + v.y;
    hi = t;
  };
  if constexpr (PARTS > 0) {
#pragma unroll
    for (int k = 0; k < PARTS; ++k) add(k);
  } else {
    const bool w = WIDE && scale[r] < 0.f;   // read beside the first pairs, which every row has
#pragma unroll 4
    for (int k = 0; k < parts; ++k) add(k);
    if (w)
      for (int k = parts; k < SV_KSPLIT; ++k) add(k);
  }
  Bout[(long long)r * ldb + c] = hi + lo;
}

// y = A x, one warp per row.  Each lane keeps a Kahan-compensated FP32 sum of
// its strided products (FP64 arithmetic is slow on this part); the 32 lane sums
// are reduced in FP64.
__global__ void gemv_f32(const float* __restrict__ A, const float* __restrict__ x, float* __restrict__ y, int rows, int cols) {
  const int row = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  float sum = 0.f, comp = 0.f;
  for (int c = lane; c < cols; c += 32) {
    const float a = A[(long long)row * cols + c], xv = x[c];
    const float p = __fmul_rn(a, xv);   // not fused into the sums below
    const float pe = fmaf(a, xv, -p);   // exact rounding error of the product
    const float yv = __fsub_rn(p, comp) + pe;
    const float t = sum + yv;
    comp = (t - sum) - yv;
    sum = t;
  }
  double acc = (double)sum - (double)comp;
  for (int o = 16; o; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) y[row] = (float)acc;
}

}  // namespace

void gemm64_nn_sub(const double* A, int lda, const double* B, int ldb, double* C, int ldc, int M, int N, int K,
                   cudaStream_t s) {
  dim3 g((N + 63) / 64, (M + 63) / 64);
  gemm64_sub<<<g, 256, 0, s>>>(A, lda, B, ldb, C, ldc, M, N, K);
}

int launch_solve(ce_ctx* ctx, const float* E, int R, float* B, int ldb, cudaStream_t s, int* launches, bool wide_rows) {
  const int n = ctx->nobs, ld = ctx->nobs_pad;
  const unsigned rb = (unsigned)(((long long)R * n + 255) / 256);
  // the FP32 form's products in pairs (the tightest error); the tensor forms, whose correction
  // error dominates, sum four hi products per compensated step (a quarter faster)
  const bool pairs = ctx->prec == CE_PREC_FP32 || ctx->prec == CE_PREC_FP64;
  if (ctx->ainv_dig) {
    int parts = 0;
    const float* scale = nullptr;   // negative: SV_KSPLIT partial pairs
    const XprodPair pair{ctx->Ainv_hi, ctx->Ainv_lo, ld, pairs ? 2 : 4};
    const int st = launch_xprod(ctx, E, n, R, n, ctx->ainv_dig, wide_rows ? &pair : nullptr, ctx->xrows, ctx->Bpart, SV_KSPLIT, &parts, &scale, s);
    if (st) return st;
    auto reduce = wide_rows ? solve_reduce<0, true> : solve_reduce<0, false>;
    reduce<<<rb, 256, 0, s>>>(ctx->Bpart, parts, scale, R, n, B, ldb);
    if (launches) *launches += 3;
    return CE_OK;
  }
  auto gemm = pairs ? solve_gemm_f32<2> : solve_gemm_f32<4>;
  gemm<<<dim3((n + SV_TC - 1) / SV_TC, (R + SV_TR - 1) / SV_TR, SV_KSPLIT), 128, 0, s>>>(E, R, n, ctx->Ainv_hi, ctx->Ainv_lo, ld,
                                                                                      ctx->Bpart);
  solve_reduce<SV_KSPLIT, false><<<rb, 256, 0, s>>>(ctx->Bpart, SV_KSPLIT, nullptr, R, n, B, ldb);
  if (launches) *launches += 2;
  return CE_OK;
}

void launch_gemv_f32(const float* Amat, const float* x, float* y, int rows, int cols, cudaStream_t s) {
  gemv_f32<<<(rows + 7) / 8, 256, 0, s>>>(Amat, x, y, rows, cols);
}

}  // namespace ce
