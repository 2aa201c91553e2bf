// The QTEA quantizer's per-layer steps on the GPU (the step before the GEMV): from full-precision
// weights W [N][K] and the curvature diagonal h = diag(H) [K] to the GEMV's inputs.
//
//  * Salient columns (Sec. 3.2): s_j = max_i W_ij^2 * h_j^2, the s largest (ties: lower column),
//    in ascending order.
//  * Ternary assignment (Sec. 3.1, Eq. 2-3): per row and group, beta = the group mean (0 without the
//    bias option), alpha = mean |W - beta|, refitted `fit_iters` times as the mean |W - beta| over
//    the nonzero codes; T = +1 where W - beta > alpha / 2, -1 where W - beta < -alpha / 2, else 0.
//  * Column-wise rescale refinement (Sec. 3.3, Eq. 6-7): `rescale_iters` rounds of
//    v_j = mean over rows with T_ij != 0 of |W_ij - beta_i| / alpha_i (1 when there are none), then
//    reassignment with the threshold v_j alpha_i / 2.
//  * alpha, beta and v rounded to binary16; the 1:4 residual on each salient column: per group of
//    four rows the row with the largest |W - (alpha v T + beta)| (ties: lower row), its position and
//    the difference in binary16.
// Every value that decides an integer is computed in float32 with the rounding of each operation
// explicit (no contraction into FMA) and every sum in index order, one thread per sum: the results
// are those of the float32 reference bit for bit. The error propagation of Sec. 3.4 is not part of
// these steps.
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "qtea_internal.h"

namespace qtea {
namespace {

constexpr int kQThreads = 256;

__device__ __forceinline__ int8_t assign(float d, float half) { return d > half ? 1 : (d < -half ? -1 : 0); }

// max_i W_ij * W_ij over a chunk of rows per block row of the grid; the squares are >= 0, so their
// bit patterns order as unsigned integers and the maximum is exact in any order.
constexpr int kQScoreRows = 128;

__global__ void __launch_bounds__(kQThreads) quant_wmax_kernel(const float* __restrict__ W, int N, int K,
                                                              unsigned* __restrict__ wmax) {
  const int j = blockIdx.x * kQThreads + threadIdx.x;
  if (j >= K) return;
  const int i0 = blockIdx.y * kQScoreRows, i1 = min(N, i0 + kQScoreRows);
  float m = 0.f;
#pragma unroll 16
  for (int i = i0; i < i1; ++i) {
    const float w = W[(size_t)i * K + j];
    m = fmaxf(m, __fmul_rn(w, w));
  }
  atomicMax(wmax + j, __float_as_uint(m));
}

// The s columns with the largest s_j = (max_i W_ij^2) * (h_j * h_j) (ties: lower column), ascending, by one
// CTA of TH threads; keys: shared memory for n_keys scores (later ones are formed again where needed). The
// scores are >= 0, so their bits order as unsigned integers (a NaN is above every number): the s-th largest
// is found bit by bit, each bit one count over all columns, and the columns above it, with the first of
// those equal to it, are written in the order of the threads' contiguous segments. (Ranking every column
// against every other took K^2 comparisons, 0.19 ms at K = 14336.)
template <int TH>
__device__ __forceinline__ void select_salient(const unsigned* __restrict__ wmax, const float* __restrict__ h, int K,
                                               int s, int32_t* __restrict__ sal, unsigned* keys, int n_keys) {
  constexpr int NW = TH / 32;
  __shared__ int warp_gt[2][NW], warp_eq[NW];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int seg = (K + TH - 1) / TH, c0 = min(K, tid * seg), c1 = min(K, c0 + seg);
  auto score = [&](int c) { return __float_as_uint(__fmul_rn(__uint_as_float(wmax[c]), __fmul_rn(h[c], h[c]))); };
  auto key = [&](int c) { return c < n_keys ? keys[c] : score(c); };
#pragma unroll 8
  for (int c = tid; c < min(K, n_keys); c += TH) keys[c] = score(c);
  __syncthreads();
  auto total = [&](unsigned t, int slot) {  // scores >= t, over all columns in any order
    int k = 0, c = tid;
#pragma unroll 16
    for (; c < min(K, n_keys); c += TH) k += keys[c] >= t ? 1 : 0;
    for (; c < K; c += TH) k += score(c) >= t ? 1 : 0;
    k = __reduce_add_sync(0xffffffffu, k);
    if (lane == 0) warp_gt[slot][warp] = k;
    __syncthreads();
    return (int)__reduce_add_sync(0xffffffffu, lane < NW ? warp_gt[slot][lane] : 0);
  };
  unsigned thr = 0u;  // the s-th largest score
  for (int bit = 31; bit >= 0; --bit) {
    const unsigned cand = thr | 1u << bit;
    if (total(cand, bit & 1) >= s) thr = cand;
  }
  const int total_gt = thr == 0xFFFFFFFFu ? 0 : total(thr + 1u, 1);
  int gt = 0, eq = 0;
  for (int c = c0; c < c1; ++c) {
    const unsigned u = key(c);
    gt += u > thr ? 1 : 0;
    eq += u == thr ? 1 : 0;
  }
  int sg = gt, se = eq;  // inclusive scans over the warp
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int a = __shfl_up_sync(0xffffffffu, sg, o), b = __shfl_up_sync(0xffffffffu, se, o);
    if (lane >= o) {
      sg += a;
      se += b;
    }
  }
  __syncthreads();  // the last total has been read
  if (lane == 31) {
    warp_gt[0][warp] = sg;
    warp_eq[warp] = se;
  }
  __syncthreads();
  int before_gt = sg - gt, before_eq = se - eq;
  for (int k = 0; k < warp; ++k) {
    before_gt += warp_gt[0][k];
    before_eq += warp_eq[k];
  }
  const int take = s - total_gt;  // columns taken of those equal to thr: the first ones
  int pos = before_gt + min(before_eq, take);
  for (int c = c0; c < c1; ++c) {
    const unsigned u = key(c);
    const bool in = u > thr || (u == thr && before_eq < take);
    before_eq += u == thr ? 1 : 0;
    if (in) sal[pos++] = c;
  }
}

constexpr int kQSelThreads = 512, kQSelKeys = 8192;
__global__ void __launch_bounds__(kQSelThreads) quant_select_kernel(const unsigned* __restrict__ wmax,
                                                                   const float* __restrict__ h, int K, int s,
                                                                   int32_t* __restrict__ sal) {
  __shared__ unsigned keys[kQSelKeys];
  select_salient<kQSelThreads>(wmax, h, K, s, sal, keys, kQSelKeys);
}

// Four (or one) consecutive floats of W into shared memory without passing through registers.
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// What the passes over W need of a (row, group): alpha, beta, the correctly rounded 1 / alpha, alpha / 2.
__device__ __forceinline__ float4 scale_record(float a, float b) { return make_float4(a, b, __frcp_rn(a), __fmul_rn(a, 0.5f)); }

// Groups of 128 columns: alpha and beta of every (row, full group), and the column maxima of W^2. A warp
// takes 32 rows x one group at a time, a row per lane: the tile arrives in shared memory by 16-byte copies
// (row stride 132 words: the lanes' 16-byte reads fall in different banks), the row goes to 128 registers
// for its passes in column order, and the next tile's copies run meanwhile. A pass costs one subtraction
// or comparison and one addition per value; |w - beta| is kept from the second pass on. No codes are
// written: they follow from W, alpha, beta and v, which the later passes read anyway. Bound: the reads of
// W and the chains of additions (12 warps per SM), about evenly. Measured (4096 x 14336, with the maxima,
// 235 MB of W): 51 us; with the maxima as a pass of their own, codes written and integer counts 70 + 35.
constexpr int kQFitWarps = 4;
constexpr int kQFitStride = 132;

__global__ void __launch_bounds__(kQFitWarps * 32, 3) quant_fit128_kernel(const float* __restrict__ W, int N, int K, int G,
                                                                          int n_groups, int row_lanes, int vec, int bias,
                                                                          int fit_iters, float4* __restrict__ ab,
                                                                          unsigned* __restrict__ wmax) {
  extern __shared__ __align__(16) float fit_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int id = blockIdx.x * kQFitWarps + warp, g = id % n_groups, r0 = id / n_groups;
  float* tl = fit_smem + warp * 32 * kQFitStride;
  const int row_blocks = (N + 31) / 32;
  if (r0 >= row_lanes) return;
  const float* base = W + (size_t)g * 128;
  auto fetch = [&](int rb) {  // rows past N: the last row again (never stored)
    for (int r = 0; r < 32; ++r) {
      const float* src = base + (size_t)min(rb * 32 + r, N - 1) * K;
      float* dst = tl + r * kQFitStride;
      if (vec) {
        cp_async16(dst + 4 * lane, src + 4 * lane);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) cp_async4(dst + lane + 32 * k, src + lane + 32 * k);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (r0 < row_blocks) fetch(r0);
  float4 cm = make_float4(0.f, 0.f, 0.f, 0.f);  // largest |w| of columns 4 lane .. 4 lane + 3
  for (int rb = r0; rb < row_blocks; rb += row_lanes) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    if (wmax) {
#pragma unroll 8
      for (int r = 0; r < 32; ++r) {
        const float4 t = *reinterpret_cast<const float4*>(tl + r * kQFitStride + 4 * lane);
        cm.x = fmaxf(cm.x, fabsf(t.x));
        cm.y = fmaxf(cm.y, fabsf(t.y));
        cm.z = fmaxf(cm.z, fabsf(t.z));
        cm.w = fmaxf(cm.w, fabsf(t.w));
      }
    }
    float w[128];
#pragma unroll
    for (int c = 0; c < 32; ++c) {
      const float4 t = *reinterpret_cast<const float4*>(tl + lane * kQFitStride + 4 * c);
      w[4 * c] = t.x;
      w[4 * c + 1] = t.y;
      w[4 * c + 2] = t.z;
      w[4 * c + 3] = t.w;
    }
    __syncwarp();  // every lane has read the tile
    if (rb + row_lanes < row_blocks) fetch(rb + row_lanes);
    float b = 0.f;
    if (bias) {
      float acc = 0.f;
#pragma unroll
      for (int c = 0; c < 128; ++c) acc = __fadd_rn(acc, w[c]);
      b = __fdiv_rn(acc, 128.f);
    }
    float acc = 0.f;
#pragma unroll
    for (int c = 0; c < 128; ++c) {
      w[c] = fabsf(__fsub_rn(w[c], b));
      acc = __fadd_rn(acc, w[c]);
    }
    float a = __fdiv_rn(acc, 128.f);
    for (int it = 0; it < fit_iters; ++it) {
      const float half = __fmul_rn(a, 0.5f);  // >= 0: d > half or d < -half is |d| > half
      float num = 0.f, cnt = 0.f;  // a count in fp32 is exact and leaves the logic pipe the comparisons alone
#pragma unroll
      for (int c = 0; c < 128; ++c)
        if (w[c] > half) {
          num = __fadd_rn(num, w[c]);
          cnt = __fadd_rn(cnt, 1.f);
        }
      if (cnt > 0.f) a = __fdiv_rn(num, cnt);
    }
    const int i = rb * 32 + lane;
    if (i < N) ab[(size_t)i * G + g] = scale_record(a, b);
  }
  if (wmax && r0 < row_blocks) {  // max of the rounded squares = the rounded square of the largest |w|
    const float m[4] = {cm.x, cm.y, cm.z, cm.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) atomicMax(wmax + g * 128 + 4 * lane + k, __float_as_uint(__fmul_rn(m[k], m[k])));
  }
}

// A last group of fewer than 128 columns (or a matrix of at most 128): one warp per 32 rows, the tile in
// shared memory (row stride 129 words: lane l's row starts in bank l), each lane's passes in column order.
constexpr int kQTailStride = 129;

__global__ void __launch_bounds__(32) quant_fit_tail_kernel(const float* __restrict__ W, int N, int K, int c0, int n, int G,
                                                           int gi, int bias, int fit_iters, float4* __restrict__ ab,
                                                           unsigned* __restrict__ wmax) {
  __shared__ float tl[32 * kQTailStride];
  const int lane = threadIdx.x, rb = blockIdx.x;
  const int rows = min(32, N - rb * 32);
#pragma unroll 8
  for (int r = 0; r < rows; ++r)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int c = lane + 32 * k;
      if (c < n) tl[r * kQTailStride + c] = W[(size_t)(rb * 32 + r) * K + c0 + c];
    }
  __syncwarp();
  if (wmax)
    for (int c = lane; c < n; c += 32) {
      float m = 0.f;
      for (int r = 0; r < rows; ++r) m = fmaxf(m, fabsf(tl[r * kQTailStride + c]));
      atomicMax(wmax + c0 + c, __float_as_uint(__fmul_rn(m, m)));
    }
  if (lane >= rows) return;
  const float* w = tl + lane * kQTailStride;
  const float fn = (float)n;
  float b = 0.f;
  if (bias) {
    float acc = 0.f;
    for (int c = 0; c < n; ++c) acc = __fadd_rn(acc, w[c]);
    b = __fdiv_rn(acc, fn);
  }
  float acc = 0.f;
  for (int c = 0; c < n; ++c) acc = __fadd_rn(acc, fabsf(__fsub_rn(w[c], b)));
  float a = __fdiv_rn(acc, fn);
  for (int it = 0; it < fit_iters; ++it) {
    const float half = __fmul_rn(a, 0.5f);
    float num = 0.f;
    int cnt = 0;
    for (int c = 0; c < n; ++c) {
      const float d = fabsf(__fsub_rn(w[c], b));
      if (d > half) {
        num = __fadd_rn(num, d);
        ++cnt;
      }
    }
    if (cnt > 0) a = __fdiv_rn(num, (float)cnt);
  }
  ab[(size_t)(rb * 32 + lane) * G + gi] = scale_record(a, b);
}

// ---------------------------------------------------------------- sums in index order by one warp
// A sum of n float32 terms in index order is a chain of n additions (4 cycles each). The two kernels below
// give each chain a lane of an adding warp that does nothing but read terms and add, and let the other
// warps form the terms of the next tile meanwhile; a term that does not count is +0, which leaves a sum
// of non-negative terms (started at +0) as it is, so the chain has no branch, and the counts are taken by
// the warps that form the terms. Two buffers of terms in shared memory, a barrier per tile; four terms of
// a lane lie side by side (16-byte reads and writes), W arrives by asynchronous copies two or three tiles
// ahead (one tile ahead through registers left 2.2 TB/s of W, and 2700 cycles per 240 additions).
constexpr int kQSumWarps = 16;                 // warp 0 adds (a CTA's warps, 8 in the smaller column sums)
constexpr int kQSumPer = 16;                   // rows (or columns) of a tile per forming warp

// Adds 16 n terms to acc: four terms at p, the next four `stride` floats on; the next 16 read ahead.
__device__ __forceinline__ float add_terms(const float* p, int stride, int n, float acc) {
  auto load = [&](float4 (&t)[4], int i) {
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] = *reinterpret_cast<const float4*>(p + (4 * i + k) * stride);
  };
  auto add = [&](const float4 (&t)[4]) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      acc = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc, t[k].x), t[k].y), t[k].z), t[k].w);
  };
  float4 t[4], u[4];
  if (n > 0) load(t, 0);
  int i = 0;
  for (; i + 2 <= n; i += 2) {
    load(u, i + 1);
    add(t);
    if (i + 2 < n) load(t, i + 2);
    add(u);
  }
  if (i < n) add(t);
  return acc;
}

// d / a for a in [2^-40, 2^40] and d in [2^-81, 2^60], y = the correctly rounded 1 / a: q = RN(d y) is within two ulps; the
// remainder d - q a is exact in one FMA, so each correction leaves the quotient correctly rounded but for
// the error of y times the remainder. The second correction starts within one ulp, where the result is the
// correctly rounded quotient (P. Markstein, IBM J. Res. Dev. 34 (1), 1990, theorem on the final step).
__device__ __forceinline__ float divide(float d, float a, float y) {
  float q = __fmul_rn(d, y);
  q = __fmaf_rn(__fmaf_rn(-q, a, d), y, q);
  return __fmaf_rn(__fmaf_rn(-q, a, d), y, q);
}

// v_j = (sum over rows with T_ij != 0, in row order, of |W_ij - beta| / alpha) / count, kept when the count
// is 0; T follows from W, alpha, beta and the v of the round before (`first`: 1): |W - beta| > v alpha / 2.
// One CTA per 32 columns. A forming warp copies its own 16 rows of each tile, and their scales, into its own
// ring, so that only the terms need a barrier; a lane takes two columns of eight rows. Where alpha and v
// lie in [2^-40, 2^40], v alpha / 2 = v (alpha / 2) and a term that counts has |W - beta| above 2^-81, so
// divide() holds below 2^60; the rest is done again with the general operations. The first CTA of a launch
// with s > 0 selects the salient columns instead, beside the sums. 16 warps where there is a CTA per SM at
// most (the chain of additions bounds, 4 cycles a row if it had its issue slots alone; measured 11.6 at 4096 x 4096:
// three forming warps share the adding warp's scheduler), 8 and two CTAs per SM above (shared memory: a third lacks
// 1.4 KB). Measured per round: 60
// us at 4096 x 14336 (235 MB of W: 3.9 TB/s), 23 us at 4096 x 4096; with W and alpha, beta read through
// registers a tile ahead, a library division per term and one column per lane 111 and 47 us. The whole
// quantizer (groups of 128 with beta, four refits, two rounds, s = 3 % of K) 837 -> 249 us at 4096 x 14336.
template <int WARPS>
struct QColSmem {
  static constexpr int kStages = WARPS == 8 ? 3 : 4, kTile = (WARPS - 1) * kQSumPer;
  float w[kStages][kTile][32];
  float term[2][kTile / 4][32][4];
  float4 scale[kStages][kTile];
};

// Two of the smaller CTAs fit in an SM's 228 KB (1 KB of each is the system's; counts and the selection's sums are static);
// their registers are kept to what three would have, 80: with more, 247.6 -> 251.2 us for the quantizer at 4096 x 14336.
static_assert(2 * (sizeof(QColSmem<8>) + 1024 + 512) <= 228 * 1024, "two CTAs per SM");

template <int WARPS>
__global__ void __launch_bounds__(WARPS * 32, WARPS == 8 ? 3 : 1) quant_colsum_kernel(
    const float* __restrict__ W, const float4* __restrict__ ab, int N, int K, int group, int G, int vec, int first,
    float* __restrict__ v, const unsigned* __restrict__ wmax, const float* __restrict__ h, int s,
    int32_t* __restrict__ sal) {
  using Smem = QColSmem<WARPS>;
  constexpr int TILE = Smem::kTile, STAGES = Smem::kStages;
  extern __shared__ __align__(16) unsigned char col_smem[];
  Smem& sm = *reinterpret_cast<Smem*>(col_smem);
  __shared__ int counts[32];
  if (s > 0 && blockIdx.x == 0) {
    select_salient<WARPS * 32>(wmax, h, K, s, sal, reinterpret_cast<unsigned*>(col_smem), (int)(sizeof(Smem) / 4));
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int j0 = ((int)blockIdx.x - (s > 0 ? 1 : 0)) * 32;
  const int g0 = j0 / group;  // groups are K or 128 columns: one per CTA
  const int n_tiles = (N + TILE - 1) / TILE;
  const int wr = (warp - 1) * kQSumPer;            // the warp's rows of a tile
  const int c = 2 * (lane & 15), r0 = 8 * (lane >> 4);  // the lane's columns, and first row, of these
  float vj[2];
  bool v_odd = false;
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    vj[q] = first || j0 + c + q >= K ? 1.f : v[j0 + c + q];
    v_odd = v_odd || !(vj[q] >= 0x1p-40f && vj[q] <= 0x1p40f);
  }
  float acc = 0.f;
  int cnt[2] = {0, 0};
  const int lr = vec ? lane >> 3 : 0, le = vec ? 4 * (lane & 7) : lane;  // the lane's place in four rows (one)
  const float* src = W + (size_t)(wr + lr) * K + j0 + le;
  const float4* ssrc = ab + (size_t)(wr + lane) * G + g0;
  const size_t row4 = 4 * (size_t)K, tile_w = (size_t)TILE * K, tile_s = (size_t)TILE * G;
  const bool col_in = j0 + le < K;  // K % 4 == 0: a vector lies wholly inside or past the row
  int left = N - wr, fill = 0;      // rows from the warp's first in the next tile, its stage
  auto issue = [&]() {
    if (left > 0) {
      const float* p = src;
      if (vec) {
#pragma unroll
        for (int i = 0; i < kQSumPer / 4; ++i, p += row4)
          if (4 * i + lr < left && col_in) cp_async16(&sm.w[fill][wr + 4 * i + lr][le], p);
      } else {
#pragma unroll 4
        for (int r = 0; r < kQSumPer; ++r, p += K)
          if (r < left && col_in) cp_async4(&sm.w[fill][wr + r][lane], p);
      }
      if (lane < kQSumPer && lane < left) cp_async16(&sm.scale[fill][wr + lane], ssrc);
      left -= TILE;
      src += tile_w;
      ssrc += tile_s;
      fill = fill + 1 == STAGES ? 0 : fill + 1;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (threadIdx.x < 32) counts[threadIdx.x] = 0;
  if (warp > 0)
    for (int k = 0; k < STAGES - 1; ++k) issue();
  int st = 0;
  for (int k = 0; k <= n_tiles; ++k) {
    if (warp == 0) {
      if (k > 0) acc = add_terms(&sm.term[(k - 1) & 1][0][lane][0], 128, TILE / 16, acc);
    } else if (k < n_tiles) {
      asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
      __syncwarp();
      const int rows = N - k * TILE - wr - r0;
      const float4* sc = &sm.scale[st][wr + r0];
      const float* w = &sm.w[st][wr + r0][c];
      float4* out = reinterpret_cast<float4*>(sm.term[k & 1][(wr + r0) / 4][c]);
      bool odd = v_odd;
      float dmax = 0.f, amin = 1.f, amax = 1.f;
#pragma unroll
      for (int r4 = 0; r4 < 2; ++r4) {
        float t[2][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = 4 * r4 + i;
          const float4 f = sc[r];
          const float2 x = *reinterpret_cast<const float2*>(w + r * 32);
          amin = fminf(amin, f.x);
          amax = fmaxf(amax, f.x);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const float d = fabsf(__fsub_rn(q ? x.y : x.x, f.y));
            const bool on = r < rows && d > __fmul_rn(vj[q], f.w);
            dmax = fmaxf(dmax, d);
            t[q][i] = on ? divide(d, f.x, f.z) : 0.f;
            cnt[q] += on ? 1 : 0;
          }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) out[32 * r4 + q] = make_float4(t[q][0], t[q][1], t[q][2], t[q][3]);
      }
      odd = odd || !(dmax <= 0x1p60f && amin >= 0x1p-40f && amax <= 0x1p40f);
      if (odd) {  // again with the general operations (rows past N may hold anything)
        for (int r = 0; r < min(rows, 8); ++r) {
          const float4 f = sc[r];
          for (int q = 0; q < 2; ++q) {
            const float d = fabsf(__fsub_rn(w[r * 32 + q], f.y));
            const bool on = d > __fmul_rn(__fmul_rn(vj[q], f.x), 0.5f);
            cnt[q] += (on ? 1 : 0) - (d > __fmul_rn(vj[q], f.w) ? 1 : 0);
            reinterpret_cast<float*>(out + 32 * (r >> 2) + q)[r & 3] = on ? __fdiv_rn(d, f.x) : 0.f;
          }
        }
      }
      __syncwarp();  // the warp has read the stage
      issue();
      st = st + 1 == STAGES ? 0 : st + 1;
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (warp > 0)
#pragma unroll
    for (int q = 0; q < 2; ++q) atomicAdd(&counts[c + q], cnt[q]);
  __syncthreads();
  if (warp == 0 && j0 + lane < K) {
    if (counts[lane] > 0) v[j0 + lane] = __fdiv_rn(acc, (float)counts[lane]);
    else if (first) v[j0 + lane] = 1.f;
  }
}

// One scale group per row, wider than 128 columns: beta (the row's mean), alpha (mean |W - beta|) and its
// refits, each a sum over the row in column order. One CTA per 32 rows, a row per lane of the adding warp.
// The other warps copy tiles of W (32 rows x 240 columns) into a ring of four by 16-byte (4-byte, where
// rows are not whole aligned vectors) copies and write the terms transposed, four columns of a row side by
// side. The chain of K additions per pass bounds it (and, close behind, forming the terms). Measured (4096 x
// 4096, no beta, four refits): 76 us, 7.6 cycles per addition; the whole quantizer 4409 us with one thread per
// row, 161 now.
constexpr int kQRowTile = 240;                 // columns of a tile: 16 per forming warp
constexpr int kQRowStride = 136;               // floats from four columns' terms to the next four's: rows x 4 + 8
constexpr int kQRowStages = 4;

struct QRowSmem {
  float w[kQRowStages][32][kQRowTile];
  float term[2][kQRowTile / 4][kQRowStride];
  float beta[32], half[32];
  int count[32];
};

__global__ void __launch_bounds__(kQSumWarps * 32, 1) quant_fit_rows_kernel(const float* __restrict__ W, int N, int K, int vec,
                                                                           int bias, int fit_iters,
                                                                           float4* __restrict__ ab) {
  extern __shared__ __align__(16) unsigned char row_smem[];
  QRowSmem& sm = *reinterpret_cast<QRowSmem*>(row_smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int i0 = blockIdx.x * 32, rows = min(32, N - i0);
  const int n_tiles = (K + kQRowTile - 1) / kQRowTile;
  const int first = bias ? 0 : 1, total = (2 + fit_iters - first) * n_tiles;  // tiles over all passes
  static_assert(kQRowTile == (kQSumWarps - 1) * 16, "16 columns of a tile per forming warp");
  const int c4 = (warp - 1) * 4 + (lane & 3), sub = lane >> 2;  // the lane's four columns; rows sub, sub + 8, ...
  const int pt = threadIdx.x - 32;
  if (warp == 0) {
    sm.beta[lane] = 0.f;
    sm.half[lane] = 0.f;
    sm.count[lane] = 0;
  }
  // copies of the next tile of the sequence of all passes' tiles; a thread's places in a tile do not change
  int left = total, c0 = 0, fill = 0;
  auto issue = [&]() {
    if (left > 0) {
      --left;
      float(*dst)[kQRowTile] = sm.w[fill];
      const float* src = W + (size_t)i0 * K + c0;
      const int n = K - c0;
      if (vec) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // 32 rows of 60 vectors over 480 threads
          const int e = pt + i * (kQSumWarps - 1) * 32, r = e / (kQRowTile / 4), c = 4 * (e - r * (kQRowTile / 4));
          if (r < rows && c < n) cp_async16(&dst[r][c], src + (size_t)r * K + c);
        }
      } else {
        for (int e = pt; e < rows * kQRowTile; e += (kQSumWarps - 1) * 32) {
          const int r = e / kQRowTile, c = e - r * kQRowTile;
          if (c < n) cp_async4(&dst[r][c], src + (size_t)r * K + c);
        }
      }
      c0 = c0 + kQRowTile < K ? c0 + kQRowTile : 0;
      fill = fill + 1 == kQRowStages ? 0 : fill + 1;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (warp > 0)
    for (int t = 0; t < kQRowStages - 1; ++t) issue();
  __syncthreads();
  float a = 0.f, b = 0.f;
  int stage = 0;
  for (int pass = first; pass < 2 + fit_iters; ++pass) {  // 0: mean, 1: mean |W - beta|, then refits
    float acc = 0.f;
    int cnt[4] = {0, 0, 0, 0};
    float be[4], half[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      be[r] = sm.beta[8 * r + sub];
      half[r] = sm.half[8 * r + sub];
    }
    for (int k = 0; k <= n_tiles; ++k) {
      if (warp == 0) {
        if (k > 0) {
          const float* p = &sm.term[(k - 1) & 1][0][4 * lane];
          const int n = min(kQRowTile, K - (k - 1) * kQRowTile);
          acc = add_terms(p, kQRowStride, n >> 4, acc);
          for (int c = n & ~15; c < n; ++c) acc = __fadd_rn(acc, p[(c >> 2) * kQRowStride + (c & 3)]);
        }
      } else if (k < n_tiles) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kQRowStages - 2) : "memory");
        asm volatile("bar.sync 1, %0;" ::"n"((kQSumWarps - 1) * 32) : "memory");  // every thread's copies of tile t
        const float(*w)[kQRowTile] = sm.w[stage];
        const int valid = K - k * kQRowTile - 4 * c4;  // columns from the lane's first
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const int i = 8 * r + sub;
          const float4 x4 = *reinterpret_cast<const float4*>(&w[i][4 * c4]);
          float x[4] = {x4.x, x4.y, x4.z, x4.w};
          if (pass > 0) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              x[q] = fabsf(__fsub_rn(x[q], be[r]));
              if (pass > 1) {
                const bool on = q < valid && x[q] > half[r];
                x[q] = on ? x[q] : 0.f;
                cnt[r] += on ? 1 : 0;
              }
            }
          }
          *reinterpret_cast<float4*>(&sm.term[k & 1][c4][4 * i]) = make_float4(x[0], x[1], x[2], x[3]);
        }
        issue();  // into the stage of the tile before, which all had read at the barrier
        stage = stage + 1 == kQRowStages ? 0 : stage + 1;
      }
      __syncthreads();
    }
    if (warp > 0 && pass > 1) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        int c = cnt[r];  // over the four lanes of the row
        c += __shfl_xor_sync(0xffffffffu, c, 1);
        c += __shfl_xor_sync(0xffffffffu, c, 2);
        if ((lane & 3) == 0) atomicAdd(&sm.count[8 * r + sub], c);
      }
    }
    __syncthreads();
    if (warp == 0) {
      if (pass == 0) b = __fdiv_rn(acc, (float)K);
      else if (pass == 1) a = __fdiv_rn(acc, (float)K);
      else if (sm.count[lane] > 0) a = __fdiv_rn(acc, (float)sm.count[lane]);
      sm.beta[lane] = b;
      sm.half[lane] = __fmul_rn(a, 0.5f);
      sm.count[lane] = 0;
    }
    __syncthreads();
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  if (warp == 0 && lane < rows) ab[i0 + lane] = scale_record(a, b);
}

__global__ void quant_fill_kernel(float* __restrict__ v, int K) {
  const int j = blockIdx.x * kQThreads + threadIdx.x;
  if (j < K) v[j] = 1.f;
}

// The outputs that follow from W, alpha, beta and v, one launch. Of every 64 rows first the CTAs that write
// the codes, then those of the residual, whose scattered reads of W then hit L2; the rounding comes last.
//  * residual: a thread per (group of four rows, salient column): T from W against v alpha / 2, W^ from the
//    binary16 alpha, beta and v, the row with the largest |W - W^| (ties: lower row), its position and the
//    difference in binary16; four lanes share a byte of positions.
//  * rounding: alpha, beta (pairs with bias) and v in binary16.
//  * codes: T_ij = nearest of {-v_j alpha, 0, +v_j alpha} to W_ij - beta. With K % 4 == 0 a thread takes four
//    columns (one 16-byte load of W, one 4-byte store of codes; the four share a scale group) of
//    kQAssignRows rows, all loads first; otherwise one column.
constexpr int kQAssignRows = 8, kQFinalRows = 64;

struct QFinal {
  const float* W;
  const float4* ab;
  const float* v;
  const int32_t* sal;
  int8_t* T;
  uint16_t *row_scale, *col_scale, *rvals;
  uint8_t* ridx;
  int N, K, group, G, s, bias;
  long long NG;
  unsigned res_blocks, col_blocks, row_blocks;  // CTAs of 64 rows' residual, of a row of codes; 64-row blocks
};

template <bool VEC>
__global__ void __launch_bounds__(kQThreads) quant_final_kernel(const QFinal p) {
  const int N = p.N, K = p.K, G = p.G;
  const unsigned code_blocks = p.col_blocks * (kQFinalRows / kQAssignRows), per_rows = code_blocks + p.res_blocks;
  const unsigned rows64 = blockIdx.x / per_rows;
  unsigned blk = blockIdx.x - rows64 * per_rows;
  if (rows64 < p.row_blocks && blk >= code_blocks) {
    const int s = p.s, s4 = (s + 3) & ~3;
    const int idx = (int)((blk - code_blocks) * kQThreads + threadIdx.x), ql = idx / s4, c = idx - ql * s4;
    const int q = (int)rows64 * (kQFinalRows / 4) + ql;
    const bool in = ql < kQFinalRows / 4 && q < N / 4;
    uint32_t bits = 0;
    if (in && c < s) {
      const int j = p.sal[c], g = j / p.group;
      float w[4];
      float4 sc[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        w[r] = p.W[(size_t)(4 * q + r) * K + j];
        sc[r] = p.ab[(size_t)(4 * q + r) * G + g];
      }
      const float v = p.v[j], vh = __half2float(__float2half_rn(v));
      int best = 0;
      float best_abs = -1.f, best_r = 0.f;
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const int t = assign(__fsub_rn(w[r], sc[r].y), __fmul_rn(__fmul_rn(v, sc[r].x), 0.5f));
        const float a = __half2float(__float2half_rn(sc[r].x)), b = p.bias ? __half2float(__float2half_rn(sc[r].y)) : 0.f;
        const float d = __fsub_rn(w[r], __fadd_rn(__fmul_rn(__fmul_rn(a, vh), (float)t), b));
        if (fabsf(d) > best_abs) {
          best_abs = fabsf(d);
          best = r;
          best_r = d;
        }
      }
      p.rvals[(size_t)q * s + c] = __half_as_ushort(__float2half_rn(best_r));
      bits = (uint32_t)best << (2 * (c & 3));
    }
    // the four entries of a byte: neighbouring lanes (s4 and the CTA are multiples of four)
    bits |= __shfl_xor_sync(0xffffffffu, bits, 1);
    bits |= __shfl_xor_sync(0xffffffffu, bits, 2);
    if (in && (c & 3) == 0) p.ridx[(size_t)q * (s4 >> 2) + (c >> 2)] = (uint8_t)bits;
    return;
  }
  if (rows64 >= p.row_blocks) {
    const long long idx = ((long long)blockIdx.x - (long long)p.row_blocks * per_rows) * kQThreads + threadIdx.x;
    if (idx < p.NG) {
      const float4 sc = p.ab[idx];
      if (p.bias) {
        p.row_scale[2 * (size_t)idx] = __half_as_ushort(__float2half_rn(sc.x));
        p.row_scale[2 * (size_t)idx + 1] = __half_as_ushort(__float2half_rn(sc.y));
      } else {
        p.row_scale[idx] = __half_as_ushort(__float2half_rn(sc.x));
      }
    }
    if (idx < K) p.col_scale[idx] = __half_as_ushort(__float2half_rn(p.v[idx]));
    return;
  }
  constexpr int per = VEC ? 4 : 1;
  const unsigned rb = blk / p.col_blocks;
  const int j = ((int)(blk - rb * p.col_blocks) * kQThreads + (int)threadIdx.x) * per;
  const int i0 = (int)rows64 * kQFinalRows + (int)rb * kQAssignRows;
  if (j >= K || i0 >= N) return;
  const int g = j / p.group;
  float vj[per];
#pragma unroll
  for (int q = 0; q < per; ++q) vj[q] = p.v[j + q];
  float w[kQAssignRows][per];
  float2 sc[kQAssignRows];
#pragma unroll
  for (int r = 0; r < kQAssignRows; ++r) {
    const int i = min(i0 + r, N - 1);
    const float* src = p.W + (size_t)i * K + j;
    if constexpr (VEC) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(src));
      w[r][0] = t.x; w[r][1] = t.y; w[r][2] = t.z; w[r][3] = t.w;
    } else {
      w[r][0] = *src;
    }
    sc[r] = __ldg(reinterpret_cast<const float2*>(p.ab + (size_t)i * G + g));
  }
#pragma unroll
  for (int r = 0; r < kQAssignRows; ++r) {
    if (i0 + r >= N) break;
    uint32_t packed = 0;
#pragma unroll
    for (int q = 0; q < per; ++q)
      packed |= (uint32_t)(uint8_t)assign(__fsub_rn(w[r][q], sc[r].y), __fmul_rn(__fmul_rn(vj[q], sc[r].x), 0.5f))
                << (8 * q);
    int8_t* dst = p.T + (size_t)(i0 + r) * K + j;
    if constexpr (VEC) *reinterpret_cast<uint32_t*>(dst) = packed;
    else *dst = (int8_t)packed;
  }
}

inline unsigned blocks(long long n, int per) { return (unsigned)((n + per - 1) / per); }

constexpr size_t kQFitSmem = (size_t)kQFitWarps * 32 * kQFitStride * sizeof(float);

// Above the default 48 KB of dynamic shared memory: opted in once per device (an attribute of the function
// on the device that is current), as is the SM count.
struct QuantDevice {
  bool ready;
  int sm_count;
};
cudaError_t quant_device(QuantDevice* out) {
  constexpr int kMaxDevices = 64;
  static QuantDevice devs[kMaxDevices];
  static std::mutex mu;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!devs[dev].ready) {
    e = cudaDeviceGetAttribute(&devs[dev].sm_count, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(quant_fit128_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kQFitSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(quant_colsum_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)sizeof(QColSmem<8>));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(quant_colsum_kernel<kQSumWarps>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)sizeof(QColSmem<kQSumWarps>));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(quant_fit_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(QRowSmem));
    if (e != cudaSuccess) return e;
    devs[dev].ready = true;
  }
  *out = devs[dev];
  return cudaSuccess;
}

}  // namespace

cudaError_t launch_quantize(const QuantArgs& a, cudaStream_t st) {
  QuantDevice dev;
  cudaError_t e = quant_device(&dev);
  if (e != cudaSuccess) return e;
  const int G = (a.K + a.group - 1) / a.group;
  const long long NG = (long long)a.N * G;
  // scratch: the scale records [N][G], v [K] (rounded up to 4 words), wmax [K]
  char* scratch = nullptr;
  const size_t kv = ((size_t)a.K + 3) & ~(size_t)3;
  e = cudaMallocAsync(&scratch, sizeof(float4) * (size_t)NG + 4 * (kv + (size_t)a.K), st);
  if (e != cudaSuccess) return e;
  float4* ab = reinterpret_cast<float4*>(scratch);
  float* v = reinterpret_cast<float*>(ab + NG);  // 16-byte aligned
  unsigned* wmax = reinterpret_cast<unsigned*>(v + kv);
  const unsigned kb = blocks(a.K, kQThreads);
  const bool w16 = a.K % 4 == 0 && (reinterpret_cast<uintptr_t>(a.W) & 15) == 0;  // rows of aligned 16-byte vectors
  if (a.s > 0) e = cudaMemsetAsync(wmax, 0, sizeof(unsigned) * (size_t)a.K, st);
  if (e == cudaSuccess) {
    unsigned* wm = a.s > 0 ? wmax : nullptr;
    if (a.group > 128) {  // one group per row
      if (wm) quant_wmax_kernel<<<dim3(kb, blocks(a.N, kQScoreRows)), kQThreads, 0, st>>>(a.W, a.N, a.K, wm);
      quant_fit_rows_kernel<<<blocks(a.N, 32), kQSumWarps * 32, sizeof(QRowSmem), st>>>(a.W, a.N, a.K, w16 ? 1 : 0, a.bias,
                                                                                       a.fit_iters, ab);
    } else {
      const int full = a.group == 128 ? a.K / 128 : 0, tail = a.K - 128 * full;
      if (full > 0) {
        // three CTAs of four warps per SM; every warp keeps one group and walks down the rows
        const int want = std::max(1, 3 * kQFitWarps * dev.sm_count / full);
        const int lanes = std::min(want, (int)blocks(a.N, 32));
        quant_fit128_kernel<<<blocks((long long)full * lanes, kQFitWarps), kQFitWarps * 32, kQFitSmem, st>>>(
            a.W, a.N, a.K, G, full, lanes, w16 ? 1 : 0, a.bias, a.fit_iters, ab, wm);
      }
      if (tail > 0)
        quant_fit_tail_kernel<<<blocks(a.N, 32), 32, 0, st>>>(a.W, a.N, a.K, 128 * full, tail, G, G - 1, a.bias,
                                                              a.fit_iters, ab, wm);
    }
    const unsigned cols = blocks(a.K, 32);
    if (a.rescale_iters == 0) {
      quant_fill_kernel<<<kb, kQThreads, 0, st>>>(v, a.K);
      if (wm) quant_select_kernel<<<1, kQSelThreads, 0, st>>>(wmax, a.h, a.K, a.s, a.sal);
    }
    for (int it = 0; it < a.rescale_iters; ++it) {
      const int s = it == 0 ? a.s : 0;  // the first round's launch selects the salient columns beside its sums
      const unsigned grid = cols + (s > 0 ? 1u : 0u);
      if ((int)grid <= dev.sm_count)
        quant_colsum_kernel<kQSumWarps><<<grid, kQSumWarps * 32, sizeof(QColSmem<kQSumWarps>), st>>>(
            a.W, ab, a.N, a.K, a.group, G, w16, it == 0, v, wmax, a.h, s, a.sal);
      else
        quant_colsum_kernel<8><<<grid, 8 * 32, sizeof(QColSmem<8>), st>>>(a.W, ab, a.N, a.K, a.group, G, w16, it == 0, v,
                                                                         wmax, a.h, s, a.sal);
    }
    const bool vec = w16 && (reinterpret_cast<uintptr_t>(a.codes) & 3) == 0;
    QFinal f;
    f.W = a.W;
    f.ab = ab;
    f.v = v;
    f.sal = a.sal;
    f.T = a.codes;
    f.row_scale = a.row_scale;
    f.col_scale = a.col_scale;
    f.rvals = a.rvals;
    f.ridx = a.ridx;
    f.N = a.N;
    f.K = a.K;
    f.group = a.group;
    f.G = G;
    f.s = a.s;
    f.bias = a.bias;
    f.NG = NG;
    f.res_blocks = a.s > 0 ? blocks((long long)(kQFinalRows / 4) * ((a.s + 3) & ~3), kQThreads) : 0u;
    f.col_blocks = blocks(vec ? a.K / 4 : a.K, kQThreads);
    f.row_blocks = blocks(a.N, kQFinalRows);
    // at most 2^14 x (8 x 2^8 + 2^12) + 2^20 x 2^9 / 2^8 CTAs: below 2^31
    const unsigned grid = f.row_blocks * (f.col_blocks * (kQFinalRows / kQAssignRows) + f.res_blocks) +
                          blocks(NG > a.K ? NG : a.K, kQThreads);
    if (vec) quant_final_kernel<true><<<grid, kQThreads, 0, st>>>(f);
    else quant_final_kernel<false><<<grid, kQThreads, 0, st>>>(f);
    e = cudaGetLastError();
  }
  const cudaError_t f = cudaFreeAsync(scratch, st);
  return e != cudaSuccess ? e : f;
}

}  // namespace qtea
