// B = E A^-1 on the tensor cores at the accuracy of FP32 output rounding: the solve of
// Eq. (condmvn) and the products of the closed-form standard errors.
//
// Every row of the symmetric matrix (an FP32 pair hi + lo) and of E is scaled by a power of
// two to |x| < 1 and cut into signed 8-bit digits, x = sum_t q_t 2^-(7 + 8 t): five for the
// matrix (to 2^-40), four for E (exact for values down to 2^-8 of the row's largest), each
// exact in bf16 with its own weight (bf16 has eight significant bits and FP32's exponents).
// Of the twenty digit products the fourteen of weight 256^-(t+u), t + u <= 4, are formed:
// those of t + u = 0, 1 and 2 in accumulators of their own, which stay exact (at most 256
// columns and three products: below 2^24 units), the rest together in a fourth, whose
// rounding lies near 2^-40.  After at most 256 columns the accumulators join a float pair
// (TwoSum of the first two, the others with the errors in the low part).
// Rows of E whose values span too many binades for that (kWideRatio: a bad station, a sparse or
// decaying right-hand side) take the FP32 products of the pair instead, tile by tile in the same
// kernel once the digits are done: a launch of its own for them cost every call 6.5 us.
// The matrix needs its 40 bits: the residuals of real data are smooth, A^-1 E cancels, and
// the correction K_go B amplifies what is left.  At n = 10000 (condition 10^4) a matrix cut
// at 2^-32 leaves 4e-4 in the draw, at 2^-40 8e-7; the FP32 CUDA-core form (compensated sums,
// 4 to 5.5 FP32 operations per useful multiply-add) leaves 9e-6.
//
// Bound: the tensor pipe (14 bf16 products), the single lane that issues them, and the
// operands' way through L2 (10 bytes per matrix element).  n = 4500, R = 100: 0.385 ms (the
// FP32 form) -> 0.053 ms; n = 2000, R = 100: 84 -> 17 us.  Below n = 1800 (kXprodMin) its
// fixed cost (digits, launch, tensor-memory set-up: 11 us for any small n) exceeds the FP32
// form's time at small R (n = 1000: 13 us at R = 8 against 8).  The whole solve in FP32 and in
// digits: n = 1800, R = 1: 30.1 and 30.0 us, R = 4: 29.0 and 33.1; n = 1900, R = 16: 35.3 and
// 33.2; n = 2000, R = 8: 32.8 and 33.9, R = 100: 100 and 38; n = 2500, R = 1: 38.4 and 38.4.
// The line is drawn by n alone, never by R: a realization's result must not depend on how
// many others are solved with it.
// One block per SM: a loader lane (bulk copies of the matrix's digit planes into a ring, of
// E's into two buffers), an MMA lane, eight epilogue warps that keep the running pairs in
// registers.  Work items: 128 rows of the matrix x up to 128 rows of E x a part of the
// columns, so that a small system still fills the SMs; the parts' pairs are added in a fixed
// order by solve_reduce.
#include <algorithm>

#include "ce_common.cuh"
#include "ce_internal.h"
#include "ce_solve_tile.cuh"
#include "ce_tc.cuh"

namespace ce {
namespace {

constexpr int kAPlanes = 5, kBPlanes = 4;   // digits of a matrix element, of an element of E
constexpr uint32_t kAPlane = 128 * 128; // bytes of one digit plane: 128 rows x 64 columns of bf16
constexpr int kUnit = 4;                // chunks of 64 columns summed in tensor memory
constexpr int kMaxRing = 8;             // digit planes of the matrix in flight
constexpr uint32_t kXprodSmem = 226 * 1024;   // most dynamic shared memory of a block
constexpr int kEpi = 8;                 // epilogue warps
// Loader, MMA and epilogue; with the FP32 products of the wide rows (CHAIN > 0) two warps more, so
// that these have three groups of 128 threads.
__host__ __device__ constexpr int xprod_threads(int chain) { return chain ? (kEpi + 4) * 32 : (kEpi + 2) * 32; }

// The digits of f, |f| < 1 (plus the low part g, |g| <= 2^-24 |f|), as bf16 bits in the
// upper halves of d: each is the remainder rounded to a multiple of 2^-(7 + 8 t).
template <int N>
__device__ __forceinline__ void digits(float f, float g, uint32_t (&d)[N]) {
  float r = f;
#pragma unroll
  for (int t = 0; t < N; ++t) {
    if (t == 3) r += g;   // |r| <= 2^-24 so far: the sum's rounding is below 2^-48
    const float magic = t == 0 ? 0x1.8p16f : (t == 1 ? 0x1.8p8f : (t == 2 ? 0x1.8p0f : (t == 3 ? 0x1.8p-8f : 0x1.8p-16f)));
    const float q = __fsub_rn(__fadd_rn(r, magic), magic);
    r = __fsub_rn(r, q);
    d[t] = __float_as_uint(q);
  }
}

// 16-byte piece of columns 8 kg .. + 7 of row r in the 128-byte-swizzled K-major layout
__device__ __forceinline__ uint32_t piece(int r, int kg) { return (uint32_t)r * 128u + ((uint32_t)(kg ^ (r & 7)) << 4); }

// e with |v| < 2^e for every |v| <= mx (mx finite, as float bits), clamped to where 2^e is a
// normal number (above 2^127 the leading digit reaches 256, which bf16 holds too).
__device__ __forceinline__ int exp_above(unsigned mx) { return max(-120, min(127, (int)(mx >> 23) - 126)); }

// A row of E is wide where some kWideSites neighbouring sites (columns) all lie more than
// kWideRatio below its largest element, or that lies outside [2^-100, 2^100).  E's digits leave
// 2^-32.8 (RMS) of the row's largest element in every element, the FP32 products' roundings 2^-25.5
// of each term: they meet where a neighbourhood lies 2^-7 below (n = 2000, one element of a normal
// row raised to f: error of B half the domain away 2.6e-8 at f = 32, 4.1e-8 at 128, 7.9e-8 at
// 256, 2e-6 at 10^4; by FP32 products 4e-8 at all).
constexpr int kWideSites = 32;
constexpr float kWideRatio = 128.f;

// kPlanes digit planes of rows [0, rows) of v (row stride ldv, n columns; lo: the low parts or
// null), one block per row.  Row r goes to row r % tile of tile r / tile: planes of tile x
// 128 bytes, kPlanes of them per chunk of 64 columns, nchunks chunks per tile.  Rows past
// `rows` and columns past n are zeros.  scale[r]: the power of two to multiply back by
// (NaN where the row is not finite), with kRange negative for a wide row.
template <int kPlanes, bool kRange>
__global__ void __launch_bounds__(256) digit_rows_kernel(const float* __restrict__ v, const float* __restrict__ lo, long long ldv,
                                                         int rows, int n, int tile, int nchunks, uint8_t* __restrict__ out,
                                                         float* __restrict__ scale) {
  __shared__ unsigned wmax[8];
  const int r = blockIdx.x;
  const bool live = r < rows;
  const float* __restrict__ src = v + (long long)(live ? r : 0) * ldv;
  const float* __restrict__ srl = lo ? lo + (long long)(live ? r : 0) * ldv : nullptr;
  unsigned mx = 0, last = 0;   // last: of the row's last kWideSites columns, which may not be a group below
  if (live) {
    if (kRange && threadIdx.x < kWideSites && threadIdx.x < n)
      last = __float_as_uint(src[max(n - kWideSites, 0) + threadIdx.x]) & 0x7fffffffu;
    for (int c = threadIdx.x; c < n; c += 256) mx = max(mx, __float_as_uint(src[c]) & 0x7fffffffu);
  }
  for (int o = 16; o; o >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (kRange) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
  }
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) mx = max(mx, wmax[w]);
  const bool finite = mx < 0x7f800000u;
  const int e = exp_above(mx);
  const float down = e == 127 ? 0x1p-127f : __uint_as_float((uint32_t)(127 - e) << 23);
  uint8_t* __restrict__ dst = out + (size_t)(r / tile) * nchunks * kPlanes * (size_t)tile * 128u;
  const int rr = r % tile;
  const float top = __uint_as_float(mx) * down;   // (1/2, 1] wherever the row is not wide for its range alone
  bool below = threadIdx.x < 32 && __uint_as_float(last) * down * kWideRatio < top;
  for (int p = threadIdx.x; p < nchunks * 8; p += 256) {   // pieces of eight columns
    uint32_t w[kPlanes][4];
    float group = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = p * 8 + j;
      const bool in = live && finite && c < n;
      uint32_t d[kPlanes];
      const float x = in ? src[c] * down : 0.f;
      if (kRange) group = fmaxf(group, fabsf(x));
      digits<kPlanes>(x, in && srl ? srl[c] * down : 0.f, d);
#pragma unroll
      for (int t = 0; t < kPlanes; ++t) {
        if (j & 1) w[t][j / 2] |= d[t] & 0xffff0000u;
        else w[t][j / 2] = d[t] >> 16;
      }
    }
    uint8_t* __restrict__ o = dst + (size_t)(p / 8) * kPlanes * (size_t)tile * 128u + piece(rr, p & 7);
#pragma unroll
    for (int t = 0; t < kPlanes; ++t)
      *reinterpret_cast<uint4*>(o + (size_t)t * tile * 128u) = make_uint4(w[t][0], w[t][1], w[t][2], w[t][3]);
    if (kRange) {   // four adjacent lanes hold a group (their pieces exist or end together)
      static_assert(kWideSites == 32, "four pieces of eight columns");
      const unsigned quad = 0xfu << (threadIdx.x & 28);
      group = fmaxf(group, __shfl_xor_sync(quad, group, 1));
      group = fmaxf(group, __shfl_xor_sync(quad, group, 2));
      below |= p / 4 * kWideSites + kWideSites <= n && group * kWideRatio < top;
    }
  }
  if (kRange) below = __syncthreads_or(below);
  if (threadIdx.x == 0) {
    const float a = __uint_as_float(mx), f = finite ? __uint_as_float((uint32_t)(127 + e) << 23) : __uint_as_float(0x7fc00000u);
    scale[r] = kRange && finite && (below || (mx > 0 && (a < 0x1p-100f || a >= 0x1p100f))) ? -f : f;
  }
}

// h += v, returning the rounding error of the sum (Knuth's TwoSum).
__device__ __forceinline__ float two_sum(float& h, float v) {
  const float t = __fadd_rn(h, v), z = __fsub_rn(t, h);
  const float e = __fadd_rn(__fsub_rn(h, __fsub_rn(t, z)), __fsub_rn(v, z));
  h = t;
  return e;
}

struct XArgs {
  const uint8_t* a;      // matrix digit planes: mtiles x nchunks x kAPlanes planes of 16 KB
  const float* ascale;
  const uint8_t* b;      // E's: nblocks x nchunks x kBPlanes planes of npad x 128 bytes
  const float* bscale;
  float2* part;          // kparts x R x n pairs
  int n, R, npad, nchunks, nblocks, kparts, cpp, items, ring;
  const float *e, *hi, *lo;   // for the wide rows (CHAIN > 0): E (R x n) and the pair
  int ld;
  uint32_t epi_wait;     // bound on the epilogue's waits for an accumulator (try_wait rounds)
  int* status;
};

// The wide rows' FP32 products, after the digits: groups of 128 threads, each with its own part
// of the block's shared memory (which no copy or product uses any more) and its own barrier.
// Bound by the FP32 pipe at 12 warps per SM: n = 4500, R = 100, every row wide 582 us in all (the
// FP32 form's own kernel, 20 warps per SM, 409); one wide row 209; none 80, as without this.
template <int CHAIN>
__device__ __forceinline__ void wide_rows(const XArgs& p, float* sm) {
  constexpr int kGroups = xprod_threads(CHAIN) / 128;
  static_assert(kGroups * SV_SMEM <= kMaxRing * kAPlane, "the smallest block (a full ring) holds the groups' tiles");
  const int group = threadIdx.x >> 7, lane = threadIdx.x & 31;
  const int ct = (p.n + SV_TC - 1) / SV_TC, per = ct * SV_KSPLIT;   // tiles of one block of rows
  const int tiles = per * ((p.R + SV_TR - 1) / SV_TR);
  for (int t = kGroups * blockIdx.x + group; t < tiles; t += kGroups * gridDim.x) {
    const int r0 = t / per * SV_TR, c = t % per;
    const uint32_t rows = __ballot_sync(0xffffffffu, r0 + lane < p.R && p.bscale[r0 + lane] < 0.f);
    if (rows == 0) continue;
    solve_tile<CHAIN>(p.e, p.R, p.n, p.hi, p.lo, p.ld, reinterpret_cast<float*>(p.part), c % ct * SV_TC, r0, c / ct, rows,
                      threadIdx.x & 127, sm + group * (SV_SMEM / sizeof(float)),
                      [&] { asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory"); });
  }
}

// CHAIN: 0, or for the wide rows the FP32 product with that many terms per compensated step.
template <int CHAIN>
__global__ void __launch_bounds__(xprod_threads(CHAIN), 1) xprod_kernel(const __grid_constant__ XArgs p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  __shared__ __align__(8) uint64_t a_full[kMaxRing], a_empty[kMaxRing], b_full[2], b_empty[2], acc_full, acc_empty, drained;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int any_wide = 0;
  const uint32_t bplane = (uint32_t)p.npad * 128u, bbuf = kBPlanes * bplane;
  if (threadIdx.x == 0) {
    for (int s = 0; s < p.ring; ++s) {
      mbar_init(smem_u32(&a_full[s]), 1);
      mbar_init(smem_u32(&a_empty[s]), 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&b_full[s]), 1);
      mbar_init(smem_u32(&b_empty[s]), 1);
    }
    mbar_init(smem_u32(&acc_full), 1);
    mbar_init(smem_u32(&acc_empty), kEpi);
    mbar_init(smem_u32(&drained), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == kEpi) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  // item -> (tile of matrix rows, block of E's rows, columns' part); parts of one tile are adjacent
  auto item_of = [&](int it, int& mt, int& nb, int& kp, int& c0, int& c1) {
    kp = it % p.kparts;
    nb = it / p.kparts % p.nblocks;
    mt = it / p.kparts / p.nblocks;
    c0 = kp * p.cpp;
    c1 = min(p.nchunks, c0 + p.cpp);
  };
  if (warp == kEpi) {
    // ------------------------------------------------------------ loader
    if (lane == 0) {
      bool ok = true;
      uint32_t nbk = 0;   // E blocks copied so far
      uint32_t slot = 0, phase = 0, na = 0;   // the ring as counters: a division per plane cost as much as the copy
      const uint32_t ring = (uint32_t)p.ring;
      for (int it = blockIdx.x; it < p.items && ok; it += gridDim.x) {
        int mt, nb, kp, c0, c1;
        item_of(it, mt, nb, kp, c0, c1);
        const uint8_t* __restrict__ pa = p.a + ((size_t)mt * p.nchunks + c0) * kAPlanes * kAPlane;
        const uint8_t* __restrict__ pb = p.b + ((size_t)nb * p.nchunks + c0) * bbuf;
        for (int c = c0; c < c1 && ok; ++c, pb += bbuf) {
          const uint32_t bs = nbk & 1u;
          if (!mbar_wait(smem_u32(&b_empty[bs]), ((nbk >> 1) & 1u) ^ 1u, &abort_flag)) { ok = false; break; }
          mbar_arrive_expect_tx(smem_u32(&b_full[bs]), bbuf);
          bulk_g2s(base + bs * bbuf, pb, bbuf, smem_u32(&b_full[bs]));
          ++nbk;
          for (int t = 0; t < kAPlanes; ++t, pa += kAPlane) {
            if (!mbar_wait(smem_u32(&a_empty[slot]), phase ^ 1u, &abort_flag)) { ok = false; break; }
            mbar_arrive_expect_tx(smem_u32(&a_full[slot]), kAPlane);
            bulk_g2s(base + 2u * bbuf + slot * kAPlane, pa, kAPlane, smem_u32(&a_full[slot]));
            ++na;
            if (++slot == ring) {
              slot = 0;
              phase ^= 1u;
            }
          }
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicExch(p.status, CE_ERR_TIMEOUT);
      }
      // copies still in flight land before the block exits
      for (uint32_t k = nbk > 2 ? nbk - 2 : 0; k < nbk; ++k)
        for (uint32_t w = 0; w < kWaitLimit && !mbar_try(smem_u32(&b_full[k & 1u]), (k >> 1) & 1u); ++w) {
        }
      for (uint32_t k = na > ring ? na - ring : 0; k < na; ++k)
        for (uint32_t w = 0; w < kWaitLimit && !mbar_try(smem_u32(&a_full[k % ring]), (k / ring) & 1u); ++w) {
        }
    }
    __syncwarp();
  } else if (warp == kEpi + 1) {
    // ------------------------------------------------------------ MMA issue
    if (lane == 0) {
      bool ok = true, issued = false;
      uint32_t nbk = 0, unit = 0, slot = 0, phase = 0;
      const uint32_t np = (uint32_t)p.npad, ring = (uint32_t)p.ring;
      const uint32_t ibase = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(128 >> 4) << 24);   // bf16 x bf16 -> FP32
      const uint32_t id1 = ibase | ((np >> 3) << 17), id2 = ibase | ((2u * np >> 3) << 17);
      const uint32_t acc1 = tmem + np, acc2 = tmem + 2u * np, acc3 = tmem + 3u * np;
      for (int it = blockIdx.x; it < p.items && ok; it += gridDim.x) {
        int mt, nb, kp, c0, c1;
        item_of(it, mt, nb, kp, c0, c1);
        for (int c = c0; c < c1 && ok; ++c) {
          const bool first = (c - c0) % kUnit == 0;
          if (first) {
            if (!mbar_wait(smem_u32(&acc_empty), (unit & 1u) ^ 1u, &abort_flag)) { ok = false; break; }
            tc_fence_after();
          }
          const uint32_t bs = nbk & 1u;
          if (!mbar_wait(smem_u32(&b_full[bs]), (nbk >> 1) & 1u, &abort_flag)) { ok = false; break; }
          ++nbk;
          const uint32_t sb = base + bs * bbuf;
          const uint64_t b0 = sw128_desc(sb), b1 = sw128_desc(sb + bplane), b2 = sw128_desc(sb + 2u * bplane),
                         b3 = sw128_desc(sb + 3u * bplane);
#pragma unroll
          for (int t = 0; t < kAPlanes; ++t) {
            if (ok) ok = mbar_wait(smem_u32(&a_full[slot]), phase, &abort_flag);
            if (ok) {
              tc_fence_after();
              const uint64_t a = sw128_desc(base + 2u * bbuf + slot * kAPlane);
              issued = true;
              // digit t of the matrix times digits u <= min(3, 4 - t) of E into accumulator
              // min(t + u, 3); two adjacent planes of E (adjacent rows) into two adjacent
              // accumulators are one product of 2 Npad columns
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {   // 16 columns each
                const uint64_t o = 2u * kk;
                const uint32_t acc = (first && kk == 0) ? 0u : 1u;
                if (t == 0) {
                  mma_issue<KIND_BF16>(tmem, a + o, b0 + o, id2, acc);
                  mma_issue<KIND_BF16>(acc2, a + o, b2 + o, id2, acc);
                } else if (t == 1) {
                  mma_issue<KIND_BF16>(acc1, a + o, b0 + o, id2, 1u);
                  mma_issue<KIND_BF16>(acc3, a + o, b2 + o, id1, 1u);
                  mma_issue<KIND_BF16>(acc3, a + o, b3 + o, id1, 1u);
                } else if (t == 2) {
                  mma_issue<KIND_BF16>(acc2, a + o, b0 + o, id2, 1u);
                  mma_issue<KIND_BF16>(acc3, a + o, b2 + o, id1, 1u);
                } else {
                  mma_issue<KIND_BF16>(acc3, a + o, b0 + o, id1, 1u);
                  if (t == 3) mma_issue<KIND_BF16>(acc3, a + o, b1 + o, id1, 1u);
                }
              }
              mma_commit(smem_u32(&a_empty[slot]));
              if (++slot == ring) {
                slot = 0;
                phase ^= 1u;
              }
            }
          }
          if (!ok) break;
          mma_commit(smem_u32(&b_empty[bs]));
          if ((c - c0) % kUnit == kUnit - 1 || c + 1 == c1) {
            mma_commit(smem_u32(&acc_full));
            ++unit;
          }
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicExch(p.status, CE_ERR_TIMEOUT);
      }
      if (issued) {   // all tensor-core work of this block has finished before the memory is freed
        mma_commit(smem_u32(&drained));
        for (uint32_t w = 0; w < kWaitLimit && !mbar_try(smem_u32(&drained), 0u); ++w) {
        }
      }
    }
    __syncwarp();
  } else if (warp < kEpi) {
    // ------------------------------------------------------------ epilogue
    // thread: one row of the matrix tile, half of E's rows (columns of the accumulators)
    const int q = warp & 3, half = warp >> 2;
    const int ncol = p.npad / 2;   // a multiple of 8
    const uint32_t lanes = (uint32_t)(32 * q) << 16;
    uint32_t unit = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < p.items && ok; it += gridDim.x) {
      int mt, nb, kp, c0, c1;
      item_of(it, mt, nb, kp, c0, c1);
      const int units = (c1 - c0 + kUnit - 1) / kUnit;
      const int i = mt * 128 + 32 * q + lane;
      float hi[64], lo[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) hi[j] = lo[j] = 0.f;
      for (int u = 0; u < units; ++u, ++unit) {
        const bool got = mbar_wait(smem_u32(&acc_full), unit & 1u, &abort_flag, p.epi_wait);
        if (!__all_sync(0xffffffffu, got)) {
          abort_flag = 1;
          if (lane == 0) atomicExch(p.status, CE_ERR_TIMEOUT);
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          if (8 * g < ncol) {
            uint32_t r0[8], r1[8], r2[8], r3[8];
            const uint32_t col = tmem + lanes + (uint32_t)(half * ncol + 8 * g);
            tmem_ld8(col, r0);
            tmem_ld8(col + (uint32_t)p.npad, r1);
            tmem_ld8(col + 2u * (uint32_t)p.npad, r2);
            tmem_ld8(col + 3u * (uint32_t)p.npad, r3);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j)   // not read before the wait
              asm volatile("" : "+r"(r0[j]), "+r"(r1[j]), "+r"(r2[j]), "+r"(r3[j]));
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              float& h = hi[8 * g + j];
              const float e0 = two_sum(h, __uint_as_float(r0[j]));
              const float e1 = two_sum(h, __uint_as_float(r1[j]));
              lo[8 * g + j] += (__uint_as_float(r2[j]) + (e0 + e1)) + __uint_as_float(r3[j]);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&acc_empty));
      }
      if (ok && i < p.n) {
        const float as = p.ascale[i];
        float2* __restrict__ dst = p.part + (size_t)kp * p.R * p.n + i;
        const int rb = nb * p.npad + half * ncol;
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          float sc[8];   // negative: a wide row, whose pairs the FP32 products write
#pragma unroll
          for (int j = 0; j < 8; ++j) sc[j] = 8 * g + j < ncol ? p.bscale[rb + 8 * g + j] : 0.f;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int row = rb + 8 * g + j;
            float h = hi[8 * g + j];   // a normalised pair: the low part is below half an ulp of the value
            const float l = two_sum(h, lo[8 * g + j]);
            if (8 * g + j < ncol && row < p.R && !(sc[j] < 0.f)) dst[(size_t)row * p.n] = make_float2(h * as * sc[j], l * as * sc[j]);
          }
        }
      }
    }
  } else {
    // ------------------------------------------------------------ are there wide rows (CHAIN > 0)
    for (int r = threadIdx.x - (kEpi + 2) * 32; r < p.R; r += 64) any_wide |= p.bscale[r] < 0.f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kEpi) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  if constexpr (CHAIN > 0) {
    if (__syncthreads_or(any_wide) && !abort_flag)
      wide_rows<CHAIN>(p, reinterpret_cast<float*>(smem_raw + (base - smem_u32(smem_raw))));
  }
}

int nchunks_of(int n) { return (n + 63) / 64; }
int mtiles_of(int n) { return (n + 127) / 128; }

}  // namespace

size_t xprod_matrix_bytes(int n) {
  return (size_t)mtiles_of(n) * nchunks_of(n) * kAPlanes * kAPlane + sizeof(float) * (size_t)mtiles_of(n) * 128;
}

void launch_xprod_matrix(const float* hi, const float* lo, int ld, int n, void* buf, cudaStream_t s) {
  const int mt = mtiles_of(n), nc = nchunks_of(n);
  uint8_t* planes = static_cast<uint8_t*>(buf);
  float* scale = reinterpret_cast<float*>(planes + (size_t)mt * nc * kAPlanes * kAPlane);
  digit_rows_kernel<kAPlanes, false><<<mt * 128, 256, 0, s>>>(hi, lo, ld, n, n, 128, nc, planes, scale);
}

namespace {
// Rows of E per block: equal blocks of at most 128, a multiple of 16.
int block_rows(int R) {
  const int nb = (R + 127) / 128;
  return ((R + nb - 1) / nb + 15) / 16 * 16;
}
}  // namespace

size_t xprod_rows_bytes(int n, int R) {
  const int np = block_rows(R), nb = (R + np - 1) / np;
  return (size_t)nb * nchunks_of(n) * kBPlanes * np * 128u + sizeof(float) * (size_t)nb * np;
}

int launch_xprod(ce_ctx* ctx, const float* E, long long lde, int R, int n, const void* matrix, const XprodPair* pair,
                 void* rows, float* part, int max_parts, int* kparts_out, const float** scale_out, cudaStream_t s) {
  const int np = block_rows(R), nb = (R + np - 1) / np, nc = nchunks_of(n), mt = mtiles_of(n);
  XArgs a;
  a.a = static_cast<const uint8_t*>(matrix);
  a.ascale = reinterpret_cast<const float*>(a.a + (size_t)mt * nc * kAPlanes * kAPlane);
  uint8_t* planes = static_cast<uint8_t*>(rows);
  float* bscale = reinterpret_cast<float*>(planes + (size_t)nb * nc * kBPlanes * np * 128u);
  a.b = planes;
  a.bscale = bscale;
  a.part = reinterpret_cast<float2*>(part);
  a.n = n;
  a.R = R;
  a.npad = np;
  a.nchunks = nc;
  a.nblocks = nb;
  a.e = E;
  a.hi = pair ? pair->hi : nullptr;
  a.lo = pair ? pair->lo : nullptr;
  a.ld = pair ? pair->ld : 0;
  a.epi_wait = ctx->wait_limit;
  a.status = ctx->dev_status;
  int nsm = 0, dev = 0;
  CE_CUDA_TRY(cudaGetDevice(&dev));
  CE_CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  // parts of the columns: the number that takes the fewest chunks on the busiest SM for one
  // block of rows, an item's start, last drain and stores counted as two chunks more.  It
  // depends on n alone, so that a realization's result does not depend on how many others
  // are solved with it.
  int kp = 1;
  long long best = -1;
  for (int k = 1; k <= std::min(nc, max_parts); ++k) {
    const int cpp = (nc + k - 1) / k;
    if ((nc + cpp - 1) / cpp != k) continue;   // an empty part
    const long long cost = ((long long)mt * k + nsm - 1) / nsm * (cpp + 2);
    if (best < 0 || cost < best) { best = cost; kp = k; }
  }
  a.cpp = (nc + kp - 1) / kp;
  a.kparts = kp;
  a.items = mt * nb * kp;
  const uint32_t bbytes = 2u * kBPlanes * (uint32_t)np * 128u;
  a.ring = std::min<int>(kMaxRing, (int)((kXprodSmem - 1024u - bbytes) / kAPlane));
  const size_t smem = (size_t)bbytes + (size_t)a.ring * kAPlane + 1024;
  auto kernel = !pair ? xprod_kernel<0> : (pair->chain == 2 ? xprod_kernel<2> : xprod_kernel<4>);
  CE_CUDA_TRY(set_max_smem(kernel, kXprodSmem));
  auto rows_kernel = pair ? digit_rows_kernel<kBPlanes, true> : digit_rows_kernel<kBPlanes, false>;
  rows_kernel<<<nb * np, 256, 0, s>>>(E, nullptr, lde, R, n, np, nc, planes, bscale);
  kernel<<<std::min(a.items, nsm), xprod_threads(pair ? pair->chain : 0), smem, s>>>(a);
  CE_CUDA_TRY(cudaGetLastError());
  *kparts_out = kp;
  if (scale_out) *scale_out = bscale;
  return CE_OK;
}

}  // namespace ce
