// The FP32 product of the solve (Eq. (condmvn)): the kernel of small systems (ce_linalg.cu), and
// inside the digit products' kernel (ce_xprod.cu) for the rows that need it.
#pragma once

#include <cstdint>

#include "ce_internal.h"

namespace ce {
namespace {

// ---------------------------------------------------------------------------
// Per-call FP32 solve: Bout (R x ldb) = E (R x n) * (Ahi + Alo) (n x n, lda).
// Block tile: 32 rows of E x 64 columns, 128 threads with 4 x 4 outputs each;
// the K range is split over KSPLIT blocks whose partial results a second
// kernel adds.  The next 32-term chunk is copied into shared memory with
// cp.async while the current one is multiplied (two buffers).
// The rows of A^-1 alternate in sign and the sum cancels heavily, and the
// correction that follows amplifies every error of B by the cancellation of
// its own sum, so each output is a compensated dot product in the manner of
// Ogita, Rump & Oishi ("Accurate sum and dot product", SIAM J. Sci. Comput.
// 26, 2005): the running sum is updated by an error-free TwoSum (Knuth) and
// its rounding errors, with the lo products, gather in a second FP32
// accumulator.  Two hi products are first joined by one FMA (a rounding
// relative to two terms, not to the running sum), which halves the work of
// the compensated form for an error a little above one rounding of B.  Each
// partial result is written as that (sum, compensation) pair; the reduction
// joins the pairs as a float pair and rounds once.
// ---------------------------------------------------------------------------
constexpr int SV_TR = 32, SV_TC = 64, SV_KC = 32, SV_KSPLIT = kSolveKSplit;
constexpr size_t SV_SMEM = sizeof(float) * 2 * (SV_TR * (SV_KC + 1) + 2 * SV_KC * SV_TC);   // two buffers of E, hi, lo

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 4- and 16-byte asynchronous copies; a copy marked invalid writes zeros and reads nothing.
__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}

// CHAIN = 2 or 4: the hi products are summed in FP32 CHAIN at a time and each such partial
// joins the running sum by an error-free TwoSum (the error kept in the compensation with
// the lo products).  The tile of rows r0 .. and columns c0 .., part kz of the K range; bit i of
// `rows`: row r0 + i is wanted (threads without one skip the products).  tid: one of 128 threads,
// which share SV_SMEM bytes at sm (16-byte aligned) and meet at barrier().
template <int CHAIN, typename Barrier>
__device__ __forceinline__ void solve_tile(const float* __restrict__ E, int R, int n, const float* __restrict__ Ahi,
                                           const float* __restrict__ Alo, int lda, float* __restrict__ part, int c0, int r0,
                                           int kz, uint32_t rows, int tid, float* sm, Barrier barrier) {
  float (*Es)[SV_TR][SV_KC + 1] = reinterpret_cast<float (*)[SV_TR][SV_KC + 1]>(sm);
  float (*Hs)[SV_KC][SV_TC] = reinterpret_cast<float (*)[SV_KC][SV_TC]>(sm + 2 * SV_TR * (SV_KC + 1));
  float (*Ls)[SV_KC][SV_TC] = Hs + 2;
  const int kper = ((n + SV_KSPLIT - 1) / SV_KSPLIT + SV_KC - 1) / SV_KC * SV_KC;
  const int kbeg = kz * kper, kend = min(n, kbeg + kper);
  const int ty = tid / 16, tx = tid % 16;
  const bool live = r0 + ty * 4 < R && (rows >> (4 * ty) & 15u);

  // Issue the copies of the chunk starting at k0 into buffer bf.
  auto load = [&](int bf, int k0) {
    for (int e = tid; e < SV_TR * SV_KC; e += 128) {
      const int rr = e / SV_KC, kk = e % SV_KC;
      const bool ok = r0 + rr < R && k0 + kk < kend;
      cp_async4(smem_addr(&Es[bf][rr][kk]), ok ? E + (long long)(r0 + rr) * n + k0 + kk : E, ok);
    }
    for (int e = tid; e < SV_KC * SV_TC / 4; e += 128) {
      const int kk = e / (SV_TC / 4), cc = (e % (SV_TC / 4)) * 4;
      const bool ok = k0 + kk < kend && c0 + cc < lda;   // lda is a multiple of 128: whole float4 in range
      const long long off = ok ? (long long)(k0 + kk) * lda + c0 + cc : 0;
      cp_async16(smem_addr(&Hs[bf][kk][cc]), Ahi + off, ok);
      cp_async16(smem_addr(&Ls[bf][kk][cc]), Alo + off, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  float sum[4][4], comp[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { sum[i][j] = 0.f; comp[i][j] = 0.f; }
  if (kbeg < kend) load(0, kbeg);
  int bf = 0;
  for (int k0 = kbeg; k0 < kend; k0 += SV_KC, bf ^= 1) {
    if (k0 + SV_KC < kend) {
      load(bf ^ 1, k0 + SV_KC);   // that buffer was released by the barrier that ended the last chunk
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    barrier();
    if (!live) {
      // none of this thread's four rows is wanted or inside R (the last row tile is partly
      // empty when R is not a multiple of SV_TR): whole warps skip the products
    } else if constexpr (CHAIN == 2) {
#pragma unroll 2
      for (int kk = 0; kk < SV_KC; kk += 2) {   // SV_KC is even; rows past kend were copied as zeros
        const float4 h4a = *reinterpret_cast<const float4*>(&Hs[bf][kk][tx * 4]);
        const float4 h4b = *reinterpret_cast<const float4*>(&Hs[bf][kk + 1][tx * 4]);
        const float4 l4a = *reinterpret_cast<const float4*>(&Ls[bf][kk][tx * 4]);
        const float4 l4b = *reinterpret_cast<const float4*>(&Ls[bf][kk + 1][tx * 4]);
        float ea[4], eb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) { ea[i] = Es[bf][ty * 4 + i][kk]; eb[i] = Es[bf][ty * 4 + i][kk + 1]; }
        const float ha[4] = {h4a.x, h4a.y, h4a.z, h4a.w}, hb[4] = {h4b.x, h4b.y, h4b.z, h4b.w};
        const float la[4] = {l4a.x, l4a.y, l4a.z, l4a.w}, lb[4] = {l4b.x, l4b.y, l4b.z, l4b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // p = e_a hi_a + e_b hi_b (one rounding); (t, es) = TwoSum(sum, p); es and the lo products to comp
            const float p = fmaf(eb[i], hb[j], __fmul_rn(ea[i], ha[j]));
            const float t = __fadd_rn(sum[i][j], p);
            const float z = __fsub_rn(t, sum[i][j]);
            const float es = __fadd_rn(__fsub_rn(sum[i][j], __fsub_rn(t, z)), __fsub_rn(p, z));
            sum[i][j] = t;
            comp[i][j] = fmaf(eb[i], lb[j], fmaf(ea[i], la[j], comp[i][j] + es));
          }
      }
    } else {
#pragma unroll 1
      for (int kk = 0; kk < SV_KC; kk += 4) {   // SV_KC is a multiple of 4; rows past kend were copied as zeros
        float hv[4][4], lv[4][4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 h4 = *reinterpret_cast<const float4*>(&Hs[bf][kk + q][tx * 4]);
          const float4 l4 = *reinterpret_cast<const float4*>(&Ls[bf][kk + q][tx * 4]);
          hv[q][0] = h4.x; hv[q][1] = h4.y; hv[q][2] = h4.z; hv[q][3] = h4.w;
          lv[q][0] = l4.x; lv[q][1] = l4.y; lv[q][2] = l4.z; lv[q][3] = l4.w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float ev[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) ev[q] = Es[bf][ty * 4 + i][kk + q];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            // p = the four hi products summed in FP32; (t, es) = TwoSum(sum, p); es and the
            // lo products to comp
            const float p = fmaf(ev[3], hv[3][j], fmaf(ev[2], hv[2][j], fmaf(ev[1], hv[1][j], __fmul_rn(ev[0], hv[0][j]))));
            const float t = __fadd_rn(sum[i][j], p);
            const float z = __fsub_rn(t, sum[i][j]);
            const float es = __fadd_rn(__fsub_rn(sum[i][j], __fsub_rn(t, z)), __fsub_rn(p, z));
            sum[i][j] = t;
            comp[i][j] = fmaf(ev[3], lv[3][j], fmaf(ev[2], lv[2][j], fmaf(ev[1], lv[1][j], fmaf(ev[0], lv[0][j], comp[i][j] + es))));
          }
        }
      }
    }
    barrier();
  }
  float2* dst = reinterpret_cast<float2*>(part) + (long long)kz * R * n;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty * 4 + i;
    if (r >= R || !(rows >> (4 * ty + i) & 1u)) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = c0 + tx * 4 + j;
      if (c < n) dst[(long long)r * n + c] = make_float2(sum[i][j], comp[i][j]);
    }
  }
}

}  // namespace
}  // namespace ce
