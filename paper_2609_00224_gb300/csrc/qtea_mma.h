// Tensor-core QTEA GEMV with staged B operands: base-3 layouts (the paper's storage, Sec. 3.5) at 1 <= M <= 16,
// 2-bit layouts at 2 <= M <= 16 (and FP8 residuals at M = 1).
//
// Computes Eq. 10 (alpha, and optionally beta, per row or per row and 128-column group) plus Eq. 11 on
// mma.sync m16n8k16 (fp16 operands, fp32 accumulation), with every operand exact:
//  * Unit of work: 256 rows x 512 columns (four 128-column blocks: 104 base-3 or 128 2-bit bytes per row). No byte
//    is decoded twice. Base-3: at M = 1 lane q of a quad decodes block q of its rows, at M >= 2 the four lanes
//    share each block's first 24 bytes, six each, and take the last two of one block each. 2-bit: lane q takes
//    every fourth word.
//  * A (weights): two base-3 bytes sit in the 16-bit halves of a register, r = 203 * byte < 2^16. The
//    top two bits of a half are then the byte's highest base-3 digit (203 / 49152 exceeds 1/243 by
//    less than 1.5e-5, and 242 * 1.5e-5 < 1/243, so no digit is ever off), and three times the other
//    fourteen bits is the same number for the next digit. ~r & 0xC000C000 turns the two digits
//    c = T + 1 into the fp16 pair 2T = -2, -0 or +2 (sign bit and top exponent bit). 2-bit codes are shifted to
//    the same two bits.
//  * B (activations): v*x is exact in fp32; times 2^E (E per chunk and batch row, so that the largest
//    is below 2^15 after the halving that 2T asks for) it is held as two fp16 columns, hi and lo, whose
//    sum hi + lo / 2^11 is exact down to 2^-28 of the chunk's largest. Products 2^24 times the chunk's mean, infinities
//    and NaN are left out and added in fp32 at the end of the tile, to the rows whose code there is not 0. Four batch
//    rows make one n8 tile. The sums are folded with 2^-E per chunk. 2-bit codes at
//    M >= 5 have v in A instead (2T * v, one exact fp16 multiply) and x in B, eight batch rows to a tile: half the
//    MMAs (at M = 16 the decoding loop alone runs at 38 weights per clock per SM, with four split tiles at 27). From
//    |v| = 2^15 on, and for infinities and NaN in x, the tile's batch row is done again in fp32.
//  * Scales: base-3 at M = 1: column pair q of the tile is non-zero only in the k slots of lane q, so that a
//    thread's accumulators hold its own block's sums; at M >= 2 the accumulators are folded per block (2-bit with
//    one scale per row: per unit). Either way alpha, and beta times the block's sum of x, are applied in fp32 (but
//    for the last two bytes of a base-3 block at M >= 2: there A is alpha * 2T, one exact fp16 multiply).
//  * Residual (Eq. 11): virtual columns, one per salient column, in steps of 16 spread over the
//    chunks: A holds the value where the stored position is the row and 0 elsewhere, B holds x.
// What bounds it: the logic pipe and the MMAs. A base-3 weight costs one and a half issued lanes of digit
// extraction, most of them on the logic pipe (64 lanes per clock per SM); that alone would run at 59
// weights per clock per SM, the MMAs of one n8 tile alone (new A registers every time: 10.9 cycles each per
// sub-partition) at 94, both together at 50, whether with 8 or 16 decoding warps. 2-bit codes: 67 and together 45
// (M <= 4). M > 4 adds MMAs, and at M = 16 the consumers decode a unit in 4700 cycles, half of
// them MMAs (sixteen consumer warps of one block, B left as it is, shifts on the multiply pipe: the same).
// Work split: the units of every problem of a group form one sequence split evenly over one persistent
// CTA per SM; a tile whose units span several CTAs is finished by the CTA holding its first unit, which
// reaches it last and adds the others' partial rows in CTA order (self-validating words, as in the
// other stream-K kernels): results do not depend on timing. 256-row units: 512-row ones left 9 % of the
// Llama3-8B layer's time to CTAs with one unit more.
// CTA: eight consumer warps (two 16-row blocks each), and two sets of four helper warps that prepare the
// units in turn, up to four ahead: the codes (TMA, or 16-byte copies where a base-3 row is not a whole number
// of 16-byte vectors), the scales and the residual (copies), and the B operand, built from x and v in
// the CTA that uses it, so that neither a pass before the kernel nor a barrier across the grid is needed.
// The helpers come first in the CTA and their global loads go out a unit ahead: one set of four, or loads
// where they are used, made the consumers wait 1000 to 4000 cycles per unit; a third set took registers from
// the decoding (34.1 us where two give 32.6).
// Measured, Llama3-8B layer in the paper's storage, seven GEMVs in one call: M = 1 82.4 -> 30.8 us (table
// lookup before), M = 4 271 -> 34.8 us (fixed-point dp4a before), M = 16 6430 -> 71 us (the general kernel).
// Qwen3-14B layer, 2-bit codes: M = 4 41.0 -> 32.8 us, M = 16 55.4 -> 53.4 us. (With the remainder in lo itself and no
// product left out, 30.4, 34.3, 71.3 and 32.3 us, and errors up to 2^-39 of a chunk's largest product: 1 to 3 % of a
// row's sum |x W^| where activations of 5e-7 stand beside one of 6e4 whose code is 0.) The same times with two activations
// of 300, or 6e4 beside N(0, 0.1); with 6e4 beside N(0, 0.001), 46, 87, 296 and 95 us. Before, the kernel of
// qtea_gemv_mb.cu, whose pass before the kernel and barrier across the grid this one does without: the barrier's
// target was part of the launch, so that replays of a captured graph did not wait (34.5 and 49.5 us, and
// other results than the direct call wherever the activations had changed).
#pragma once

#include <cuda_fp16.h>

#include "qtea_internal.h"

namespace qtea {
namespace {

// The kernel's forms: base-3 codes at M = 1 and M >= 2, 2-bit codes with v*x split in two fp16 columns
// per batch row (M <= 4, and where the launch asks for it) and with v in A and x in B (M >= 5).
enum XMode { kXDiag = 0, kXRows = 1, kXSplit2 = 2, kXV2 = 3 };


// Partial rows of split tiles are stored XOR-ed with this NaN bit pattern, so that zeroed memory
// reads as "not written yet" and every word validates itself.
constexpr uint32_t kXPartEmpty = 0x7FBADBADu;

__device__ __forceinline__ void x_mma(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y));
}
__device__ __forceinline__ void x_mma_first(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b.x), "r"(b.y), "f"(0.f));
}
__device__ __forceinline__ uint32_t x_hmul2(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("mul.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ void x_cp16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// Eight bytes, the last 8 - n of them zero (n = 8 or 0).
__device__ __forceinline__ void x_cp8(uint32_t dst, const void* src, int n) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
// Arrival on `bar` once this thread's earlier cp.async copies have landed (counted in the barrier).
__device__ __forceinline__ void x_cp_arrive(uint32_t bar) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t x_part_load(const uint32_t* p) {
  uint32_t w;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(w) : "l"(p) : "memory");
  return w;
}
__device__ __forceinline__ void x_part_store(uint32_t* p, uint32_t w) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(w) : "memory");
}

// CTA whose range contains unit u (the inverse of unit_begin_of).
__device__ __forceinline__ int x_unit_owner(long long u, long long total, int grid) {
  return (int)(((u + 1) * grid - 1) / total);
}

// A unit's problem, tile and chunk. The ceil(s / 16) steps of 16 salient entries are spread over a
// tile's chunks: chunk ch takes steps [ch nb / n, (ch + 1) nb / n), here rs and its remainder.
struct XPos {
  int p, t, ch, rs, rem;
};
__device__ __forceinline__ XPos x_pos(const XProblem* tab, int n_problems, int u) {
  int p = 0;
  while (p + 1 < n_problems && u >= tab[p + 1].unit_begin) ++p;
  const int v = u - tab[p].unit_begin, nc = tab[p].n_chunks, t = v / nc, ch = v - t * nc;
  const int e = ch * (tab[p].res_q * nc + tab[p].res_r), rs = e / nc;  // below 2 kXMaxChunks^2
  return {p, t, ch, rs, e - rs * nc};
}
// What x_next needs of the unit's problem; in registers where every unit asks for it (shared memory reads in a
// row cost a unit some 200 cycles).
struct XShape {
  int n_chunks, res_q, res_r;
};
__device__ __forceinline__ XShape x_shape(const XProblem& a) { return {a.n_chunks, a.res_q, a.res_r}; }
template <typename T>
__device__ __forceinline__ int x_res_steps(const XPos& c, const T& a) {
  return a.res_q + (c.rem + a.res_r >= a.n_chunks ? 1 : 0);
}
// The next unit of problem a, whose shape is sh; true when it belongs to the next problem.
template <typename T>
__device__ __forceinline__ bool x_next(XPos& c, const T& sh, const XProblem& a) {
  c.rs += sh.res_q;
  c.rem += sh.res_r;
  if (c.rem >= sh.n_chunks) {
    c.rem -= sh.n_chunks;
    ++c.rs;
  }
  if (++c.ch < sh.n_chunks) return false;
  c.ch = c.rs = c.rem = 0;
  if (++c.t < a.n_tiles) return false;
  c.t = 0;
  ++c.p;
  return true;
}

// ---------------------------------------------------------------- helpers

// The unit's code bytes: row r of the tile is copied from the 16-byte boundary at or below its first
// byte, so that it starts at its own offset (0 .. 14, even) in its slot of row_slot bytes. (Rows of whole
// 16-byte vectors come by TMA instead, with the same offsets, 0 or 8.)
template <int H>
__device__ __forceinline__ void x_issue_codes(const XProblem& a, const XPos& c, uint32_t dst, int row_slot,
                                              int ht) {
  const int r0 = ht >> 3, j = ht & 7;
  const int bytes = 26 * min(4, a.n_blocks - 4 * c.ch);
  const size_t start = (size_t)(c.t * kXTileRows + r0) * a.row_bytes + (size_t)c.ch * kXChunkBytes;
  const int off = (int)(start & 15);  // the same for every 8th row: 8 row_bytes is a multiple of 16
  const uint8_t* src = a.packed + (start - off) + 16 * j;
  dst += r0 * row_slot + 16 * j;
  const int rows = a.N - c.t * kXTileRows - r0;
  constexpr int kRows = H * 4;  // rows per pass
  const size_t step = (size_t)kRows * a.row_bytes;
  if (16 * j < off + bytes) {
#pragma unroll 4
    for (int r = 0; r < kXTileRows; r += kRows)
      if (r < rows) x_cp16(dst + r * row_slot, src + (size_t)(r / kRows) * step);
  }
}

// Where column c of a block goes in the B operand of a tile: bits 0 .. 13 the byte offset (without the n
// column), bits 14 and 15 an XOR on the n column, so that the builder's scattered stores fall in different
// banks. Byte c / 5 of the block holds the column as digit c % 5, extracted at level 4 - c % 5.
// DIAG: lane q decodes block q. Bytes 0 .. 23 four at a time, bytes 4u, 4u + 2 and 4u + 1, 4u + 3 in the
// halves of an even and an odd register: step 5u + level, k slots 2q, 2q + 1 (even) and 2q + 8, 2q + 9
// (odd); bytes 24 and 25 share a register whose levels fill steps 30 .. 32. The offset is without 8q.
// Else: the four lanes share a block's first 24 bytes, six each, in steps 8 block .. 8 block + 7: the first
// four as above in five steps, the last two as bytes 24 and 25 above in three. Bytes 24 and 25 of block q
// go to lane q in steps 32 .. 34 (bit 13 set). The offset is without the block.
template <bool DIAG>
__device__ __forceinline__ uint32_t x_b_offset(int c) {
  const int byte = c / 5, level = 4 - (c - 5 * byte);
  const uint32_t half_step = (uint32_t)((level >> 1) * 256 + 4 * (level & 1)), xor_n = (uint32_t)(level & 3) << 14;
  if (byte >= 24) return half_step + 2 * (byte - 24) + (DIAG ? 30 * 256 : 1u << 13);
  const int w = DIAG ? byte & 3 : byte % 6;
  const uint32_t base = DIAG ? (uint32_t)(byte >> 2) * 1280 : (uint32_t)(byte / 6) * 8;
  if (w < 4) return (base + level * 256 + 4 * (w & 1) + 2 * (w >> 1)) | xor_n;
  return base + 1280 + half_step + 2 * (w - 4);
}

__device__ __forceinline__ bool x_finite(uint16_t h) { return (h & 0x7C00u) != 0x7C00u; }

// Sixteen columns of x (rows m0, m0 + step, ...) and v per lane: columns 16 lane .. 16 lane + 15 of chunk ch, zero
// past K and from row M on.
template <int R>
struct XRows {
  uint32_t x[R][8], v[8];
};
template <int R>
__device__ __forceinline__ void x_load_rows(const XProblem& a, int ch, int m0, int step, int M, bool with_v, int lane,
                                            XRows<R>& r) {
  const int col = ch * kXChunkCols + 16 * lane;
#pragma unroll
  for (int k = -1; k < R; ++k) {
    uint32_t (&d)[8] = k < 0 ? r.v : r.x[k < 0 ? 0 : k];
    const int m = m0 + k * step;
    const uint16_t* src = k < 0 ? a.v + col : a.x + (size_t)m * a.K + col;
#pragma unroll
    for (int i = 0; i < 8; ++i) d[i] = 0u;
    if (k < 0 ? !with_v : m >= M) continue;
    if (a.xv_vec) {  // rows of whole 16-byte vectors, 16-byte aligned
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (col + 8 * i < a.K) {
          const uint4 t = __ldg(reinterpret_cast<const uint4*>(src) + i);
          d[4 * i] = t.x; d[4 * i + 1] = t.y; d[4 * i + 2] = t.z; d[4 * i + 3] = t.w;
        }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (col + i < a.K) d[i >> 1] |= (uint32_t)__ldg(src + i) << (16 * (i & 1));
    }
  }
}

// v*x as an fp16 pair: f = v*x 2^(E - 1) below 2^15 (half of 2^E, since A is 2T), hi = f rounded, lo = the
// remainder times 2^11, so that the pair is hi + lo / 2^11. f has 22 bits: above 2^-14 the pair is f itself (hi and
// the remainder's 11 bits are normal, or the remainder is a multiple of 2^-35); below, that is 2^-28 of the largest, it is
// off by 2^-36 at most, 2^(e - 50) for products below 2^(e + 1). E follows from the chunk's largest product, but no
// further from the others than keeps that error below theirs in fp32: products of 2^(e + 1) and more, infinities and
// NaN are left out of B and added by the consumers in fp32 (x_scan, x_left_out).
constexpr float kXLo = 0x1p-11f;
// The product of the two fp16 halves i (0: low), exact in fp32, and a half's addition to an fp32 sum: mixed-precision
// instructions (PTX ISA 8.6, sm_100 and up), one each where two conversions and the operation would be two or three.
__device__ __forceinline__ uint16_t x_half(uint32_t w, int i) { return (uint16_t)(w >> (16 * i)); }
__device__ __forceinline__ float x_fma16(uint16_t a, uint16_t b, float c) {
  float d;
  asm("fma.rn.f32.f16 %0, %1, %2, %3;" : "=f"(d) : "h"(a), "h"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float x_add16(uint16_t a, float c) {
  float d;
  asm("add.rn.f32.f16 %0, %1, %2;" : "=f"(d) : "h"(a), "f"(c));
  return d;
}
__device__ __forceinline__ float x_max_nan(float a, float b) {  // NaN when either is
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
// The pair of two products: hi = RN(p sc), lo = (p sc - hi) 2^11, both from p in one exact step each.
__device__ __forceinline__ void x_pair(float p0, float p1, float sc, __half2& hi, __half2& lo) {
  hi = __floats2half2_rn(p0 * sc, p1 * sc);
  const uint32_t h = *reinterpret_cast<const uint32_t*>(&hi);
  const float sc2 = sc * 2048.f;
  lo = __floats2half2_rn(x_fma16(x_half(h, 0), 0xE800u, p0 * sc2), x_fma16(x_half(h, 1), 0xE800u, p1 * sc2));  // -2048
}
// 2 |p| in the float's bits, without the sign: 0 for zero, from kXInf on infinities and NaN.
__device__ __forceinline__ uint32_t x_mag(float p) { return __float_as_uint(p) << 1; }
constexpr uint32_t kXInf = 0xFF000000u;
// f(i, product i of the lane's sixteen) of batch row m in chunk ch, read from global memory eight columns at a time: for
// what runs rarely, in functions of its own. (As part of the kernel's loops that code cost a call of one unit per CTA
// 0.3 us and the Llama3-8B layer in the paper's storage up to 6, although it never ran; at the tile's end, as calls, it
// costs three calls of small layers at M = 11 0.3 us each.)
template <typename F>
__device__ __forceinline__ void x_products(const XProblem& a, int ch, int m, int lane, const F& f) {
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int col = ch * kXChunkCols + 16 * lane + 8 * h;
    const uint16_t *x = a.x + (size_t)m * a.K + col, *v = a.v + col;
    uint4 xw = make_uint4(0u, 0u, 0u, 0u), vw = xw;
    if (a.xv_vec) {
      if (col < a.K) {
        xw = __ldg(reinterpret_cast<const uint4*>(x));
        vw = __ldg(reinterpret_cast<const uint4*>(v));
      }
    } else {
      uint32_t xs[4] = {0u, 0u, 0u, 0u}, vs[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (col + i < a.K) {
          xs[i >> 1] |= (uint32_t)__ldg(x + i) << (16 * (i & 1));
          vs[i >> 1] |= (uint32_t)__ldg(v + i) << (16 * (i & 1));
        }
      xw = make_uint4(xs[0], xs[1], xs[2], xs[3]);
      vw = make_uint4(vs[0], vs[1], vs[2], vs[3]);
    }
    const uint32_t xs[4] = {xw.x, xw.y, xw.z, xw.w}, vs[4] = {vw.x, vw.y, vw.z, vw.w};
#pragma unroll
    for (int i = 0; i < 8; ++i) f(8 * h + i, x_fma16(x_half(vs[i >> 1], i & 1), x_half(xs[i >> 1], i & 1), 0.f));
  }
}
__device__ __forceinline__ int x_lane() {
  int lane;
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
  return lane;
}
// A row's factors from e, the binade of its largest |v*x| (< 2^(e + 1)).
__device__ __forceinline__ float x_sc(int e) { return __uint_as_float((uint32_t)(127 + 14 - e) << 23); }    // 2^(E - 1)
__device__ __forceinline__ float x_fold(int e) { return __uint_as_float((uint32_t)(127 - 15 + e) << 23); }  // 2^-E
__device__ __forceinline__ uint32_t x_largest(float lmax) {  // bits of the largest |v*x| over the lanes
  return __reduce_max_sync(0xffffffffu, __float_as_uint(lmax));
}
__device__ __forceinline__ int x_binade(uint32_t amax) {  // 128 for an infinity or NaN, 0 for zero
  return amax ? (int)(amax >> 23) - 127 : 0;
}
// The row may need another E (then x_search looks): with an infinity or NaN, or unless of the lanes with columns at
// least half (rounded up) hold a product of 2^-20 of the largest, beside which an error of 2^-50 of it is nothing.
__device__ __forceinline__ bool x_maybe(uint32_t amax, float lmax, int half) {
  const uint32_t low = amax > 20u << 23 ? amax - (20u << 23) : 0u;
  return amax >= 0x7F800000u || __popc(__ballot_sync(0xffffffffu, __float_as_uint(lmax) >= low)) < half;
}

// Products left out of a row of binade e: 2^(e + 1) and more, infinities and NaN.
__device__ __forceinline__ bool x_outside(float p, int e) { return x_mag(p) >= (uint32_t)(128 + e) << 24; }
// The binade of a row, by a warp: that of its largest finite product, but at most 24 above the mean binade of those that
// are not zero. The pairs' error, 2^(e - 50), is then below 2^-26 of that mean; an fp32 sum rounds at 2^-24 of itself.
__device__ __forceinline__ int x_scan(const XProblem& a, int ch, int m, int lane, bool* rebuild) {
  float lmax = 0.f;
  int sum = 0, n = 0;
  bool inf = false;
  x_products(a, ch, m, lane, [&](int, float p) {
    const uint32_t mag = x_mag(p);
    if (mag >= kXInf) {
      inf = true;
    } else if (mag) {
      lmax = fmaxf(lmax, fabsf(p));
      sum += (int)(mag >> 24) - 127;
      ++n;
    }
  });
  const int top = x_binade(x_largest(lmax));
  sum = __reduce_add_sync(0xffffffffu, sum);
  n = __reduce_add_sync(0xffffffffu, n);
  const int e = n ? min(top, (sum >= 0 ? sum / n : -((n - 1 - sum) / n)) + 24) : 0;
  *rebuild = __any_sync(0xffffffffu, inf) || e < top;
  return e;
}
// After batch row m of a chunk has been built from its largest product: true when it has been built again with zeros in
// the places of products that are left out (layouts: x_build_row and x_build_row2).
template <bool BASE3, bool DIAG>
__device__ __noinline__ bool x_search(const XProblem& a, int ch, int m, float* fold, const uint32_t* boff, uint8_t* bt) {
  const int lane = x_lane();
  bool rebuild;
  const int e = x_scan(a, ch, m, lane, &rebuild);
  if (!rebuild) return false;
  const float sc = x_sc(e);
  const int q = lane >> 3, w = lane >> 2, n = BASE3 ? (DIAG ? 2 * q : 2 * (m & 3)) : (2 * (m & 3)) ^ (w & 3);
  uint8_t* base = bt + (BASE3 ? (DIAG ? 8 * q : (m >> 2) * kXBTileBytes + 2048 * q)
                              : (m >> 2) * kXTile2Bytes + w * 1024 + (lane & 3) * 8);
  x_products(a, ch, m, lane, [&](int i, float p) {
    uint32_t o = ((i & 7) >> 1) * 256 + 4 * (i & 1) + 2 * (i >> 3), col = (uint32_t)n;
    if (BASE3) {
      o = (boff[8 * (lane & 7) + (i >> 1)] >> (16 * (i & 1))) & 0xFFFFu;
      col ^= o >> 14;
      o = DIAG ? o & 0x3FFFu : (o & 0x1FFFu) + (o & 0x2000u ? 8192 - 2048 * q + 8 * q : 0);
    }
    __half2 hi, lo;
    x_pair(x_outside(p, e) ? 0.f : p, 0.f, sc, hi, lo);
    *reinterpret_cast<__half*>(base + o + 32 * col) = __low2half(hi);
    *reinterpret_cast<__half*>(base + o + 32 * (col ^ 1u)) = __low2half(lo);
  });
  if (lane == 0) fold[m] = x_fold(e);
  return true;
}

// One batch row's B operand of a chunk, by one warp (lane = 16 columns; boff: the block's places, two
// columns a word). True when the row may need another E. DIAG (M =
// 1): column pair q of the tile for block q, else column pair m % 4. The factor 2^-E and the blocks'
// sums of x go to fold[m] and sx[block][m].
template <bool DIAG>
__device__ __forceinline__ bool x_build_row(const uint32_t (&x)[8], const uint32_t (&v)[8], int m, const uint32_t* boff, uint8_t* bt, float* fold,
                                            float* sx, int half, int lane) {
  // v*x is exact in fp32; formed here for the largest and again below (sixteen registers fewer)
  auto product = [&](int i) { return x_fma16(x_half(v[i >> 1], i & 1), x_half(x[i >> 1], i & 1), 0.f); };
  float sum = 0.f, lmax = 0.f;
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    sum = x_add16(x_half(x[i >> 1], i & 1), sum);
    lmax = x_max_nan(lmax, fabsf(product(i)));
  }
  const uint32_t amax = x_largest(lmax);
  const int e = x_binade(amax);
  const float sc = x_sc(e);
  if (lane == 0) fold[m] = x_fold(e);
  const int q = lane >> 3, n = DIAG ? 2 * q : 2 * (m & 3);  // the lane's block, the hi column
  uint8_t* tile = bt + (DIAG ? 8 * q : (m >> 2) * kXBTileBytes + 2048 * q);
  const int tail = 8192 - 2048 * q + 8 * q;  // from there: bytes 24 and 25
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t ow = boff[8 * (lane & 7) + i];
    __half2 hi, lo;
    x_pair(product(2 * i), product(2 * i + 1), sc, hi, lo);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t o = (ow >> (16 * k)) & 0xFFFFu;
      const uint32_t lx = (uint32_t)n ^ (o >> 14);  // n even: the lo column n + 1 is n's neighbour XOR 1
      uint8_t* d = tile + (DIAG ? o & 0x3FFFu : (o & 0x1FFFu) + (o & 0x2000u ? tail : 0));
      *reinterpret_cast<__half*>(d + 32 * lx) = k ? __high2half(hi) : __low2half(hi);
      *reinterpret_cast<__half*>(d + 32 * (lx ^ 1u)) = k ? __high2half(lo) : __low2half(lo);
    }
  }
  sum += __shfl_xor_sync(0xffffffffu, sum, 1);
  sum += __shfl_xor_sync(0xffffffffu, sum, 2);
  sum += __shfl_xor_sync(0xffffffffu, sum, 4);
  if ((lane & 7) == 0) sx[16 * q + m] = sum;
  return x_maybe(amax, lmax, half);
}

// 2-bit codes: one batch row's B operand of a chunk, by one warp. The lane's 16 columns are one code word, W =
// 4w + q: step 4w + T takes its columns 2T, 2T + 8 (k slots 2q, 2q + 1) and 2T + 1, 2T + 9 (slots 2q + 8, 2q
// + 9), so a lane's part of a step is one 8-byte store. The lanes of steps 4w .. 4w + 3 are stored XOR-ed
// with 4 (w & 3). Split: columns 2 (m % 4) and + 1 of tile m / 4 hold the fp16 pair whose sum is v*x 2^E / 2;
// else column m % 8 of tile m / 8 holds x itself. SUM: the groups' sums of x too (for beta).
template <bool SPLIT, bool SUM>
__device__ __forceinline__ bool x_build_row2(const uint32_t (&x)[8], const uint32_t (&v)[8], int m, uint8_t* bt, float* fold,
                                             float* sx, int half, int lane) {
  const int q = lane & 3, w = lane >> 2, key = w & 3;
  float sum = 0.f;
  uint8_t* base = bt + (SPLIT ? m >> 2 : m >> 3) * kXTile2Bytes + w * 1024 + q * 8;
  bool maybe = false;
  if constexpr (SPLIT) {
    auto product = [&](int i) { return x_fma16(x_half(v[i >> 1], i & 1), x_half(x[i >> 1], i & 1), 0.f); };
    float lmax = 0.f;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (SUM) sum = x_add16(x_half(x[i >> 1], i & 1), sum);
      lmax = x_max_nan(lmax, fabsf(product(i)));
    }
    const uint32_t amax = x_largest(lmax);
    const int e = x_binade(amax);
    const float sc = x_sc(e);
    if (lane == 0) fold[m] = x_fold(e);
    maybe = x_maybe(amax, lmax, half);
    const int n = (2 * (m & 3)) ^ key;
#pragma unroll
    for (int T = 0; T < 4; ++T) {
      uint32_t hi[2], lo[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        __half2 h, l;
        x_pair(product(2 * T + k), product(2 * T + k + 8), sc, h, l);
        hi[k] = *reinterpret_cast<const uint32_t*>(&h);
        lo[k] = *reinterpret_cast<const uint32_t*>(&l);
      }
      *reinterpret_cast<uint2*>(base + T * 256 + 32 * n) = make_uint2(hi[0], hi[1]);
      *reinterpret_cast<uint2*>(base + T * 256 + 32 * (n ^ 1)) = make_uint2(lo[0], lo[1]);
    }
  } else {
    const int n = (m & 7) ^ key;
    if (SUM) {
#pragma unroll
      for (int i = 0; i < 16; ++i) sum += h2f((uint16_t)(x[i >> 1] >> (16 * (i & 1))));
    }
#pragma unroll
    for (int T = 0; T < 4; ++T)
      *reinterpret_cast<uint2*>(base + T * 256 + 32 * n) =
          make_uint2(__byte_perm(x[T], x[T + 4], 0x5410), __byte_perm(x[T], x[T + 4], 0x7632));
  }
  if (SUM) {
    sum += __shfl_xor_sync(0xffffffffu, sum, 1);
    sum += __shfl_xor_sync(0xffffffffu, sum, 2);
    sum += __shfl_xor_sync(0xffffffffu, sum, 4);
    if ((lane & 7) == 0) sx[16 * (lane >> 3) + m] = sum;
  }
  return maybe;
}
// v in the same order, [32 steps][4 lanes] 8-byte entries.
__device__ __forceinline__ void x_build_v(const uint32_t (&v)[8], uint8_t* vt, int lane) {
#pragma unroll
  for (int T = 0; T < 4; ++T)
    *reinterpret_cast<uint2*>(vt + ((4 * (lane >> 2) + T) * 4 + (lane & 3)) * 8) =
        make_uint2(__byte_perm(v[T], v[T + 4], 0x5410), __byte_perm(v[T], v[T + 4], 0x7632));
}

// The unit's scales as (alpha, beta) fp16 pairs [256 rows][4 blocks] (0 past the last block), by copies
// where a row's four pairs are one aligned 16-byte vector (four alphas: one 8-byte load).
template <int H>
__device__ __forceinline__ void x_stage_scales(const XProblem& a, const XPos& c, uint8_t* dst, int ht) {
  const int nb = min(4, a.n_blocks - 4 * c.ch);
#pragma unroll
  for (int k = 0; k < kXTileRows / (32 * H); ++k) {
    const int r = ht + k * 32 * H, row = c.t * kXTileRows + r;
    if (row >= a.N) {  // zero: their alphas take part in the warp's votes
      *reinterpret_cast<uint4*>(dst + r * 16) = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    if (a.scales_vec && a.bias) {
      x_cp16(smem_u32(dst + r * 16), a.scales + 2 * ((size_t)row * a.G + 4 * c.ch));
      continue;
    }
    uint32_t w[4] = {0u, 0u, 0u, 0u};
    if (a.scales_vec) {
      const uint2 v2 = __ldg(reinterpret_cast<const uint2*>(a.scales + (size_t)row * a.G + 4 * c.ch));
      w[0] = v2.x & 0xFFFFu; w[1] = v2.x >> 16; w[2] = v2.y & 0xFFFFu; w[3] = v2.y >> 16;
    } else if (a.G == 1) {
      const uint32_t ab = (uint32_t)__ldg(a.scales + (size_t)row * (a.bias ? 2 : 1)) |
                          (a.bias ? (uint32_t)__ldg(a.scales + (size_t)row * 2 + 1) << 16 : 0u);
#pragma unroll
      for (int b = 0; b < 4; ++b) w[b] = b < nb ? ab : 0u;
    } else {
#pragma unroll
      for (int b = 0; b < 4; ++b)
        if (b < nb) {
          const size_t e = (size_t)row * a.G + 4 * c.ch + b;
          w[b] = a.bias ? (uint32_t)__ldg(a.scales + 2 * e) | (uint32_t)__ldg(a.scales + 2 * e + 1) << 16
                        : (uint32_t)__ldg(a.scales + e);
        }
    }
    *reinterpret_cast<uint4*>(dst + r * 16) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// The unit's residual values as stored, 16 per (group of four rows, step) = (ht >> 1, ht & 1), zero past
// the last entry: by copies where rows are whole aligned 8-byte words.
__device__ __forceinline__ void x_stage_residual(const XProblem& a, const XPos& c, int st0, int n_steps, uint8_t* vals,
                                                 int ht) {
  const int gl = ht >> 1, k = ht & 1, grp = c.t * (kXTileRows / 4) + gl;
  if (gl >= kXTileRows / 4 || k >= n_steps || 4 * grp >= a.N) return;
  const int e0 = 16 * (st0 + k), ne = min(16, a.s - e0);
  const size_t e = (size_t)grp * a.s + e0;
  uint8_t* d = vals + gl * kXResStride + 32 * k;
  if (a.res_vec) {
    const uint8_t* src = reinterpret_cast<const uint8_t*>(a.rvals) + (a.fp8 ? e : 2 * e);
    const int n = a.fp8 ? ne : 2 * ne;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < 2 || !a.fp8) x_cp8(smem_u32(d + 8 * i), 8 * i < n ? src + 8 * i : src, 8 * i < n ? 8 : 0);
    return;
  }
  for (int i = 0; i < 16; ++i) {
    if (a.fp8) d[i] = i < ne ? __ldg(reinterpret_cast<const uint8_t*>(a.rvals) + e + i) : (uint8_t)0;
    else reinterpret_cast<uint16_t*>(d)[i] = i < ne ? __ldg(reinterpret_cast<const uint16_t*>(a.rvals) + e + i) : (uint16_t)0;
  }
}

// The position bytes of the same entries (packed where they are stored: the loads are not waited for here).
struct XPosBytes {
  uint32_t b[4];
};
__device__ __forceinline__ void x_load_pos(const XProblem& a, const XPos& c, int st0, int n_steps, int ht, XPosBytes& p) {
  const int k = ht & 1, grp = c.t * (kXTileRows / 4) + (ht >> 1);
  const int rs = (a.s + 3) >> 2, b0 = 4 * (st0 + k);
  const bool in = ht < kXTileRows / 2 && k < n_steps && 4 * grp < a.N;
  const uint8_t* pp = a.ridx + (size_t)grp * rs + b0;
#pragma unroll
  for (int i = 0; i < 4; ++i) p.b[i] = in && b0 + i < rs ? (uint32_t)__ldg(pp + i) : 0u;
}

// The unit's salient column of this lane's entry, as stored.
__device__ __forceinline__ bool x_has_sal(const XProblem& a, int st0, int n_steps, int lane) {
  return lane < 16 * n_steps && 16 * st0 + lane < a.s;
}
__device__ __forceinline__ uint16_t x_at_sal(const XProblem& a, int m, int col) {
  return __ldg(a.x + (size_t)m * a.K + (col < 0 ? 0 : (col >= a.K ? a.K - 1 : col)));
}

// ---------------------------------------------------------------- consumers

// Two FP8 E4M3 bytes as an fp16 pair (exact).
__device__ __forceinline__ uint32_t x_e4m3x2(uint32_t b) {
  uint32_t d;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(d) : "h"((uint16_t)b));
  return d;
}

// One residual step: A = the row's values at the entries whose stored position is the row: the position byte of
// four entries, XOR-ed with the row's position in every field, indexes a table of the four 16-bit lanes' masks
// (a field that becomes zero keeps its lane). Forming the masks here took four times the logic instructions,
// 0.15 of a 2-bit unit's time.
__device__ __forceinline__ uint2 x_mask(uint32_t d) {
  return make_uint2((d & 3u ? 0u : 0xFFFFu) | (d & 0xCu ? 0u : 0xFFFF0000u),
                    (d & 0x30u ? 0u : 0xFFFFu) | (d & 0xC0u ? 0u : 0xFFFF0000u));
}
template <int MT, int BLK>
__device__ __forceinline__ void x_res_step(const uint8_t* vals, const uint8_t* pos, const uint8_t* rb,
                                           const uint2* mask, int step, bool fp8, int tr, int g, int q, int lane,
                                           float (&acc)[BLK][MT][4]) {
  uint2 b[MT];
#pragma unroll
  for (int j = 0; j < MT; ++j) b[j] = *reinterpret_cast<const uint2*>(rb + j * kXResBBytes + (step * 32 + lane) * 8);
#pragma unroll
  for (int k = 0; k < BLK; ++k) {
    uint32_t av[4];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gl = (tr + 16 * k + 8 * h + g) >> 2;
      uint32_t lo, hi;
      if (fp8) {
        const uint32_t w = *reinterpret_cast<const uint32_t*>(vals + gl * kXResStride + 32 * step + 4 * q);
        lo = x_e4m3x2(w & 0xFFFFu);
        hi = x_e4m3x2(w >> 16);
      } else {
        const uint2 w = *reinterpret_cast<const uint2*>(vals + gl * kXResStride + 32 * step + 8 * q);
        lo = w.x;
        hi = w.y;
      }
      const uint2 m = mask[(uint32_t)pos[gl * 8 + 4 * step + q] ^ ((uint32_t)(g & 3) * 0x55u)];
      av[h] = lo & m.x;
      av[2 + h] = hi & m.y;
    }
#pragma unroll
    for (int j = 0; j < MT; ++j) x_mma(acc[k][j], av[0], av[1], av[2], av[3], b[j]);
  }
}

// A pair of code bytes decoded digit by digit, the highest first (see the header). IMAD: the digits are
// taken out for the next step as r - (r & 0xC000C000) = r + digit() - 0xC000C000 on the multiply pipe
// instead of a mask on the logic pipe, which is the busier one: with every other register that way the
// decode alone runs at 50.7 weights per clock per SM against 47.9.
template <bool IMAD>
struct XDigits {
  uint32_t r;
  __device__ __forceinline__ void start(uint32_t bytes) { r = bytes * 203u; }  // a byte in each half
  __device__ __forceinline__ uint32_t digit() const { return ~r & 0xC000C000u; }
  __device__ __forceinline__ void next() {
    if (IMAD) {
      uint32_t t;
      asm("mad.lo.u32 %0, %1, 3, %2;" : "=r"(t) : "r"(digit()), "r"(0u - 3u * 0xC000C000u));
      asm("mad.lo.u32 %0, %1, 3, %2;" : "=r"(r) : "r"(r), "r"(t));
    } else {
      r = (r & 0x3FFF3FFFu) * 3u;
    }
  }
};

// M = 1: the unit's 33 steps for the warp's 16-row blocks, lane q's weights all of block q. codes: the
// stage's rows, from the aligned word that holds the lane's first byte; sh: 0, or 16 when that byte is the
// word's third. sum[.][0 / 1]: rows g, g + 8 over block q. (2T leaves 11-bit products, which the tensor
// core's sums lose little of; alpha in A would make them 22 bits, truncated at every step: 6.7e-7.)
template <int BLK>
__device__ __forceinline__ void x_decode_diag(const uint8_t* codes, int row_slot, int sh, const uint8_t* bt, int lane,
                                              float (&sum)[BLK][2]) {
  constexpr int R = 2 * BLK;  // the thread's rows: 8 apart
  const int stride = 8 * row_slot;
  float acc[2][BLK][4];  // the steps alternate between two sets
#pragma unroll
  for (int k = 0; k < 2 * BLK; ++k)
#pragma unroll
    for (int z = 0; z < 4; ++z) acc[k & 1][k >> 1][z] = 0.f;
  uint32_t w[R];
#pragma unroll
  for (int r = 0; r < R; ++r) w[r] = *reinterpret_cast<const uint32_t*>(codes + r * stride);
#pragma unroll 2
  for (int u = 0; u < 6; ++u) {
    XDigits<false> e[R];
    XDigits<true> o[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t nx = *reinterpret_cast<const uint32_t*>(codes + r * stride + 4 * u + 4);
      const uint32_t x = __funnelshift_r(w[r], nx, sh);
      w[r] = nx;
      e[r].start(x & 0x00FF00FFu);
      o[r].start(__byte_perm(x, 0u, 0x4341));
    }
#pragma unroll
    for (int l = 0; l < 5; ++l) {
      const uint2 b = *reinterpret_cast<const uint2*>(bt + (5 * u + l) * 256 + (lane ^ (4 * (l & 3))) * 8);
#pragma unroll
      for (int k = 0; k < BLK; ++k)
        x_mma(acc[(u + l) & 1][k], e[2 * k].digit(), e[2 * k + 1].digit(), o[2 * k].digit(), o[2 * k + 1].digit(), b);
      if (l < 4) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          e[r].next();
          o[r].next();
        }
      }
    }
  }
  XDigits<false> e[R];
#pragma unroll
  for (int r = 0; r < R; ++r) e[r].start(__byte_perm(w[r] >> sh, 0u, 0x4140));
#pragma unroll
  for (int l = 0; l < 5; l += 2) {
    const uint2 b = *reinterpret_cast<const uint2*>(bt + ((30 + l / 2) * 32 + lane) * 8);
    uint32_t a0[R], a1[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      a0[r] = e[r].digit();
      e[r].next();
      a1[r] = l < 4 ? e[r].digit() : 0u;
      e[r].next();
    }
#pragma unroll
    for (int k = 0; k < BLK; ++k) x_mma(acc[(l >> 1) & 1][k], a0[2 * k], a0[2 * k + 1], a1[2 * k], a1[2 * k + 1], b);
  }
#pragma unroll
  for (int k = 0; k < BLK; ++k) {
    sum[k][0] = fmaf(acc[0][k][1] + acc[1][k][1], kXLo, acc[0][k][0] + acc[1][k][0]);
    sum[k][1] = fmaf(acc[0][k][3] + acc[1][k][3], kXLo, acc[0][k][2] + acc[1][k][2]);
  }
}

// Alphas (fp16 bits) whose 2T alpha could be infinite, and those that may not be divided by 4.
__device__ __forceinline__ bool x_big(uint32_t h) { return (h & 0x7FFFu) >= 0x7400u; }
__device__ __forceinline__ bool x_tiny(uint32_t h) { return (h & 0x7FFFu) - 1u < 0x0C00u - 1u; }  // below 2^-12, not 0

// M >= 2: the unit's 35 steps. The four lanes share each block (six bytes each, one accumulation of eight
// steps, scaled by the rows' alpha in fp32: run += alpha_b 2^-E sum + beta_b sum_b(x)); the blocks' last
// two bytes go to one lane each and carry alpha in A (a sixteenth of the columns, three steps; tiny: the lane has
// alphas there that are left out). row: the
// offset of the thread's first row in the stage; off: of the unit in the row.
template <int MT, int BLK>
__device__ __forceinline__ void x_decode_rows(const uint8_t* row, int off, int row_slot, const uint8_t* bt,
                                              const uint8_t* sc, const float* fold, const float* sx, bool bias,
                                              int q, int lane, bool& tiny, float (&run)[BLK][MT][2]) {
  constexpr int R = 2 * BLK;
  const int stride = 8 * row_slot;
  // the unit's sum on its own before it joins the tile's: 28 additions in a row instead of 112 for K = 14336
  float acc[BLK][MT][4], part[BLK][MT][2];
#pragma unroll
  for (int k = 0; k < BLK; ++k)
#pragma unroll
    for (int j = 0; j < MT; ++j) part[k][j][0] = part[k][j][1] = 0.f;
#pragma unroll 1
  for (int blk = 0; blk < 4; ++blk) {
    const int o0 = off + 26 * blk + 6 * q, sh = 8 * (o0 & 2);
    const uint8_t* wp = row + (o0 & ~3);
    const uint8_t* bb = bt + blk * 2048;
    XDigits<false> e[R], y[R];
    XDigits<true> o[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t w0 = *reinterpret_cast<const uint32_t*>(wp + r * stride);
      const uint32_t w1 = *reinterpret_cast<const uint32_t*>(wp + r * stride + 4);
      const uint32_t x = __funnelshift_r(w0, w1, sh);
      e[r].start(x & 0x00FF00FFu);
      o[r].start(__byte_perm(x, 0u, 0x4341));
      y[r].start(__byte_perm(w1 >> sh, 0u, 0x4140));
    }
#pragma unroll
    for (int l = 0; l < 5; ++l) {
      uint2 b[MT];
#pragma unroll
      for (int j = 0; j < MT; ++j)
        b[j] = *reinterpret_cast<const uint2*>(bb + j * kXBTileBytes + l * 256 + (lane ^ (4 * (l & 3))) * 8);
#pragma unroll
      for (int k = 0; k < BLK; ++k) {
        const uint32_t a0 = e[2 * k].digit(), a1 = e[2 * k + 1].digit(), a2 = o[2 * k].digit(), a3 = o[2 * k + 1].digit();
#pragma unroll
        for (int j = 0; j < MT; ++j) {
          if (l == 0) x_mma_first(acc[k][j], a0, a1, a2, a3, b[j]);
          else x_mma(acc[k][j], a0, a1, a2, a3, b[j]);
        }
      }
      if (l < 4) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          e[r].next();
          o[r].next();
        }
      }
    }
#pragma unroll
    for (int l = 0; l < 5; l += 2) {
      uint2 b[MT];
#pragma unroll
      for (int j = 0; j < MT; ++j)
        b[j] = *reinterpret_cast<const uint2*>(bb + j * kXBTileBytes + (5 + l / 2) * 256 + lane * 8);
      uint32_t a0[R], a1[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a0[r] = y[r].digit();
        y[r].next();
        a1[r] = l < 4 ? y[r].digit() : 0u;
        y[r].next();
      }
#pragma unroll
      for (int k = 0; k < BLK; ++k)
#pragma unroll
        for (int j = 0; j < MT; ++j) x_mma(acc[k][j], a0[2 * k], a0[2 * k + 1], a1[2 * k], a1[2 * k + 1], b[j]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const uint32_t ab = *reinterpret_cast<const uint32_t*>(sc + r * 128 + 4 * blk);
      const float al = h2f((uint16_t)ab), be = h2f((uint16_t)(ab >> 16));
#pragma unroll
      for (int j = 0; j < MT; ++j) {
        float& t = part[r >> 1][j][r & 1];
        const float* a2 = &acc[r >> 1][j][2 * (r & 1)];
        t = fmaf(al, fmaf(a2[1], kXLo, a2[0]) * fold[4 * j + q], t);
        if (bias) t = fmaf(be, sx[16 * blk + 4 * j + q], t);
      }
    }
  }
  // bytes 24 and 25 of block q; alpha * 2T must stay finite: with some |alpha| >= 2^14 the warp takes alpha / 4, but for
  // alphas that could lose bits that way (x_tiny), which are added at the end of the tile (x_left_out)
  uint32_t al[R];
  bool big = false;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    al[r] = __byte_perm(*reinterpret_cast<const uint32_t*>(sc + r * 128 + 4 * q), 0u, 0x1010);
    big = big || x_big(al[r]);
  }
  float up = 1.f;
  if (__any_sync(0xffffffffu, big)) {
    up = 4.f;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      tiny = tiny || x_tiny(al[r]);
      al[r] = x_tiny(al[r]) ? 0u : x_hmul2(al[r], 0x34003400u);
    }
  }
  XDigits<false> y[R];
  const int o0 = off + 26 * q + 24;
#pragma unroll
  for (int r = 0; r < R; ++r)
    y[r].start(__byte_perm((uint32_t)*reinterpret_cast<const uint16_t*>(row + o0 + r * stride), 0u, 0x4140));
#pragma unroll
  for (int l = 0; l < 5; l += 2) {
    uint2 b[MT];
#pragma unroll
    for (int j = 0; j < MT; ++j)
      b[j] = *reinterpret_cast<const uint2*>(bt + j * kXBTileBytes + (32 + l / 2) * 256 + lane * 8);
    uint32_t a0[R], a1[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      a0[r] = x_hmul2(y[r].digit(), al[r]);
      y[r].next();
      a1[r] = l < 4 ? x_hmul2(y[r].digit(), al[r]) : 0u;
      y[r].next();
    }
#pragma unroll
    for (int k = 0; k < BLK; ++k)
#pragma unroll
      for (int j = 0; j < MT; ++j) {
        if (l == 0) x_mma_first(acc[k][j], a0[2 * k], a0[2 * k + 1], a1[2 * k], a1[2 * k + 1], b[j]);
        else x_mma(acc[k][j], a0[2 * k], a0[2 * k + 1], a1[2 * k], a1[2 * k + 1], b[j]);
      }
  }
#pragma unroll
  for (int k = 0; k < BLK; ++k)
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      const float F = fold[4 * j + q] * up;
      run[k][j][0] += fmaf(fmaf(acc[k][j][1], kXLo, acc[k][j][0]), F, part[k][j][0]);
      run[k][j][1] += fmaf(fmaf(acc[k][j][3], kXLo, acc[k][j][2]), F, part[k][j][1]);
    }
}

// 2-bit codes: A = 2T of columns i and i + 8 of a code word: shifted left by 14 - 2i, their codes c = T + 1 lie at
// bits 14-15 and 30-31, and ~w & 0xC000C000 makes each the fp16 value -2, -0 or +2.
// MUL: the shift as a multiplication by a kernel parameter (an immediate would become a shift again), which
// issues beside the logic pipe: every other register that way decodes 67 weights per clock per SM against 62
// (no gain where A is multiplied by v as well).
template <int I, bool MUL>
__device__ __forceinline__ uint32_t x_a2(uint32_t w, const XParams& P) {
  return ~(MUL && I < 7 ? w * P.shift[I] : w << (14 - 2 * I)) & 0xC000C000u;
}

// Step 4w + T (columns 2T, 2T + 8 and 2T + 1, 2T + 9 of the rows' code words c).
template <int MT, int BLK, bool SPLIT, int T>
__device__ __forceinline__ void x_step2(const uint8_t* bt, const uint8_t* vt, int w, int q, int lane,
                                        const uint32_t (&c)[2 * BLK], bool first, const XParams& P,
                                        float (&acc)[BLK][MT][4]) {
  uint2 b[MT];
  uint2 vp = make_uint2(0u, 0u);
#pragma unroll
  for (int j = 0; j < MT; ++j)
    b[j] = *reinterpret_cast<const uint2*>(bt + j * kXTile2Bytes + (4 * w + T) * 256 + (lane ^ (4 * (w & 3))) * 8);
  if (!SPLIT) vp = *reinterpret_cast<const uint2*>(vt + ((4 * w + T) * 4 + q) * 8);
#pragma unroll
  for (int k = 0; k < BLK; ++k) {
    uint32_t a0 = x_a2<2 * T, SPLIT>(c[2 * k], P), a1 = x_a2<2 * T, SPLIT>(c[2 * k + 1], P);
    uint32_t a2 = x_a2<2 * T + 1, SPLIT>(c[2 * k], P), a3 = x_a2<2 * T + 1, SPLIT>(c[2 * k + 1], P);
    if (!SPLIT) {
      a0 = x_hmul2(a0, vp.x);
      a1 = x_hmul2(a1, vp.x);
      a2 = x_hmul2(a2, vp.y);
      a3 = x_hmul2(a3, vp.y);
    }
#pragma unroll
    for (int j = 0; j < MT; ++j) {
      if (first) x_mma_first(acc[k][j], a0, a1, a2, a3, b[j]);
      else x_mma(acc[k][j], a0, a1, a2, a3, b[j]);
    }
  }
}

constexpr int kXFoldV = 2;
// The unit's 32 steps, 2-bit codes. Lane q takes word 4w + q of its rows (16-byte segment w of the row, stored
// at segment w ^ (row % 8)). SPLIT: B holds (hi, lo) of v*x 2^E / 2, folded with 2^-E; else A = 2T * v, one exact
// fp16 multiply by the pairs in vt, and B holds x. GRP: the accumulators are folded per 128-column group with
// the rows' alpha and beta of the group (staged at sc), else per unit with the row's alpha (al); with v in A,
// whose products have 22 bits, two or four times a unit. out: added to, [block]
// [tile][value]: SPLIT rows g, g + 8 of batch row 4 tile + q; else (row, batch row 8 tile + 2q + 0 / 1).
template <int MT, int BLK, bool SPLIT, bool GRP>
__device__ __forceinline__ void x_decode2(const uint8_t* codes, const uint8_t* bt, const uint8_t* vt, const uint8_t* sc,
                                          const float* fold, const float* sx, bool bias, const float (&al)[2 * BLK],
                                          int g, int q, int lane, const XParams& P,
                                          float (&out)[BLK][MT][SPLIT ? 2 : 4]) {
  constexpr int R = 2 * BLK;
  // The steps alternate between two sets of accumulators: half the chain, and MMAs that do not wait for one
  // another (14b layer, M = 16: 54.3 -> 53.2 us); with one tile and v in A one set folded twice as often is
  // faster (M = 8: 39.1 us; 40.2 with two).
  constexpr bool kTwo = SPLIT ? MT == 1 : (GRP || MT > 1);  // (split tiles beyond the first: registers)
  constexpr int kFold = GRP || !kTwo ? 2 : 4;                // words (four steps each) per fold
  float acc[2][BLK][MT][4];
#pragma unroll (MT == 1 && (SPLIT || !GRP) ? 8 : (GRP ? 2 : 4))  // registers
  for (int w = 0; w < 8; ++w) {
    uint32_t c[R];
#pragma unroll
    for (int r = 0; r < R; ++r) c[r] = *reinterpret_cast<const uint32_t*>(codes + r * 1024 + ((w ^ g) << 4));
    const bool first = w % kFold == 0;
    x_step2<MT, BLK, SPLIT, 0>(bt, vt, w, q, lane, c, first, P, acc[0]);
    x_step2<MT, BLK, SPLIT, 1>(bt, vt, w, q, lane, c, first && kTwo, P, acc[kTwo ? 1 : 0]);
    x_step2<MT, BLK, SPLIT, 2>(bt, vt, w, q, lane, c, false, P, acc[0]);
    x_step2<MT, BLK, SPLIT, 3>(bt, vt, w, q, lane, c, false, P, acc[kTwo ? 1 : 0]);
    if (w % kFold != kFold - 1) continue;
    const int blk = w >> 1;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float a1 = al[r], be = 0.f;
      if (GRP) {
        const uint32_t ab = *reinterpret_cast<const uint32_t*>(sc + r * 128 + 4 * blk);
        a1 = h2f((uint16_t)ab);
        be = h2f((uint16_t)(ab >> 16));
      }
      if (!SPLIT) a1 *= 0.5f;
#pragma unroll
      for (int j = 0; j < MT; ++j) {
        const float *d = &acc[0][r >> 1][j][2 * (r & 1)], *e = &acc[1][r >> 1][j][2 * (r & 1)];
        if constexpr (SPLIT) {
          float& t = out[r >> 1][j][r & 1];
          const float sum = (kTwo ? fmaf(d[1] + e[1], kXLo, d[0] + e[0]) : fmaf(d[1], kXLo, d[0])) * fold[4 * j + q];
          if (GRP) t += fmaf(a1, sum, bias ? be * sx[16 * blk + 4 * j + q] : 0.f);
          else t = fmaf(a1, sum, t);
        } else {
#pragma unroll
          for (int z = 0; z < 2; ++z) {
            float& t = out[r >> 1][j][2 * (r & 1) + z];
            if (GRP) t += fmaf(a1, d[z] + e[z], bias ? be * sx[16 * blk + 8 * j + 2 * q + z] : 0.f);
            else t = fmaf(a1, kTwo ? d[z] + e[z] : d[z], t);
          }
        }
      }
    }
  }
}

// What B leaves out of batch row m in chunk ch: the sum of alpha T (v*x) in fp32, and of the residual's values times
// x where x is not finite, for the thread's rows row0, row0 + 8, + 16, + 24. Everything is read from global memory
// again: two passes over the chunk to find the columns, some 500 cycles for each. Rare (an activation 2^24
// times the chunk's mean).
template <bool BASE3, bool DIAG>
__device__ __noinline__ float4 x_left_out(const XProblem& a, int ch, int m, int row0) {
  constexpr int R = 2 * kXBlocks;
  const int lane = x_lane();
  const uint16_t* xm = a.x + (size_t)m * a.K;
  bool rebuild;
  const int e = x_scan(a, ch, m, lane, &rebuild);
  uint32_t mask = 0u;
  if (rebuild)
    x_products(a, ch, m, lane, [&](int i, float p) {
      if (x_outside(p, e)) mask |= 1u << i;
    });
  float out[R];
#pragma unroll
  for (int r = 0; r < R; ++r) out[r] = 0.f;
  for (uint32_t lanes; (lanes = __ballot_sync(0xffffffffu, mask != 0u)) != 0u;) {
    const int src = __ffs((int)lanes) - 1;
    const int k = ch * kXChunkCols + 16 * src + __ffs((int)__shfl_sync(0xffffffffu, mask, src)) - 1;
    if (lane == src) mask &= mask - 1u;
    const float p = x_fma16(__ldg(a.v + k), __ldg(xm + k), 0.f);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = min(row0 + 8 * r, a.N - 1);  // rows past N: never written
      const uint8_t* codes = a.packed + (size_t)row * a.row_bytes;
      int T;
      if (BASE3) {
        int b = __ldg(codes + 26 * (k >> 7) + (k & 127) / 5);
        for (int d = (k & 127) % 5; d > 0; --d) b /= 3;
        T = b % 3 - 1;
      } else {
        T = ((__ldg(codes + (k >> 2)) >> (2 * (k & 3))) & 3) - 1;
      }
      const size_t g = a.G == 1 ? (size_t)row : (size_t)row * a.G + (k >> 7);
      if (T) out[r] = fmaf(h2f(__ldg(a.scales + (a.bias ? 2 * g : g))), T > 0 ? p : -p, out[r]);
    }
  }
  if (BASE3 && !DIAG) {  // the last two bytes of block q where x_decode_rows left them out
    const int blk = 4 * ch + (lane & 3);
    uint16_t al[R];
    bool big = false;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = row0 + 8 * r;
      const size_t g = a.G == 1 ? (size_t)row : (size_t)row * a.G + blk;
      al[r] = row < a.N && blk < a.n_blocks ? __ldg(a.scales + (a.bias ? 2 * g : g)) : (uint16_t)0;
      big = big || x_big(al[r]);
    }
    if (__any_sync(0xffffffffu, big)) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float sum = 0.f;
        if (x_tiny(al[r])) {
          const uint8_t* codes = a.packed + (size_t)(row0 + 8 * r) * a.row_bytes + 26 * blk;
          int b = __ldg(codes + 24) + 243 * __ldg(codes + 25);
          for (int k = 128 * blk + 120; k < min(a.K, 128 * blk + 128); ++k, b /= 3) {
            const float p = x_fma16(__ldg(a.v + k), __ldg(xm + k), 0.f);
            if (!x_outside(p, e)) sum = fmaf((float)(b % 3 - 1), p, sum);  // those that B holds
          }
        }
        sum *= h2f(al[r]);
        sum += __shfl_xor_sync(0xffffffffu, sum, 1);
        out[r] += sum + __shfl_xor_sync(0xffffffffu, sum, 2);
      }
    }
  }
  const int at = ch * (a.res_q * a.n_chunks + a.res_r), st0 = at / a.n_chunks;
  const int n_steps = a.res_q + (at - st0 * a.n_chunks + a.res_r >= a.n_chunks ? 1 : 0);
  uint16_t xs = 0;
  if (x_has_sal(a, st0, n_steps, lane)) xs = x_at_sal(a, m, __ldg(a.sal + 16 * st0 + lane));
  for (uint32_t lanes = __ballot_sync(0xffffffffu, !x_finite(xs)); lanes; lanes &= lanes - 1u) {
    const int src = __ffs((int)lanes) - 1, c = 16 * st0 + src;
    const float xe = h2f((uint16_t)__shfl_sync(0xffffffffu, (uint32_t)xs, src));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = min(row0 + 8 * r, a.N - 1), grp = row >> 2;
      if (((__ldg(a.ridx + (size_t)grp * ((a.s + 3) >> 2) + (c >> 2)) >> (2 * (c & 3))) & 3) != (row & 3)) continue;
      const size_t i = (size_t)grp * a.s + c;
      const uint16_t h = a.fp8 ? (uint16_t)x_e4m3x2(__ldg(reinterpret_cast<const uint8_t*>(a.rvals) + i))
                               : __ldg(reinterpret_cast<const uint16_t*>(a.rvals) + i);
      out[r] = fmaf(h2f(h), xe, out[r]);
    }
  }
  return make_float4(out[0], out[1], out[2], out[3]);
}

// Batch row m over chunks ch0 .. ch1 with v in A, done again in fp32 as the general kernels do, for the thread's rows row0,
// row0 + 8, + 16, + 24 (the quad's lanes take every fourth column and salient entry). For tiles that came out
// infinite or NaN: from |v| = 2^15 on 2v is no fp16 number, and an infinity or NaN in x meets every row through 0 *
// x; here it counts in the rows whose code, or residual position, it meets. Found by looking at the tile's sums, which
// costs nothing (looking at x and v as they are staged: Qwen3-14B layer, M = 16, 53.2 -> 54.7 us).
__device__ __noinline__ float4 x_again(const XProblem& a, int ch0, int ch1, int m, int row0) {
  constexpr int R = 2 * kXBlocks;
  const int q = x_lane() & 3;
  const uint16_t* xm = a.x + (size_t)m * a.K;
  const uint8_t* codes[R];
  const uint16_t* scales[R];
  float out[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int row = min(row0 + 8 * r, a.N - 1);  // rows past N: never written
    codes[r] = a.packed + (size_t)row * a.row_bytes;
    scales[r] = a.scales + (size_t)row * a.G * (a.bias ? 2 : 1);
    out[r] = 0.f;
  }
  for (int k = ch0 * kXChunkCols + q; k < min(a.K, (ch1 + 1) * kXChunkCols); k += 4) {
    const uint16_t xk = __ldg(xm + k);
    const float p = x_fma16(__ldg(a.v + k), xk, 0.f);
    const int g = a.G == 1 ? 0 : k >> 7;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int T = ((__ldg(codes[r] + (k >> 2)) >> (2 * (k & 3))) & 3) - 1;
      if (T) out[r] = fmaf(h2f(__ldg(scales[r] + (a.bias ? 2 * g : g))), T > 0 ? p : -p, out[r]);
      if (a.bias) out[r] = fmaf(h2f(__ldg(scales[r] + 2 * g + 1)), h2f(xk), out[r]);
    }
  }
  const int per = a.res_q * a.n_chunks + a.res_r;  // the chunks' salient entries: steps [ch0 per / n, (ch1 + 1) per / n)
  const int c1 = min(a.s, 16 * (int)((long long)(ch1 + 1) * per / a.n_chunks));
  for (int c = 16 * (ch0 * per / a.n_chunks) + q; c < c1; c += 4) {
    const float xc = h2f(x_at_sal(a, m, __ldg(a.sal + c)));
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = min(row0 + 8 * r, a.N - 1), grp = row >> 2;
      if (((__ldg(a.ridx + (size_t)grp * ((a.s + 3) >> 2) + (c >> 2)) >> (2 * (c & 3))) & 3) != (row & 3)) continue;
      const size_t i = (size_t)grp * a.s + c;
      const uint16_t h = a.fp8 ? (uint16_t)x_e4m3x2(__ldg(reinterpret_cast<const uint8_t*>(a.rvals) + i))
                               : __ldg(reinterpret_cast<const uint16_t*>(a.rvals) + i);
      out[r] = fmaf(h2f(h), xc, out[r]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    out[r] += __shfl_xor_sync(0xffffffffu, out[r], 1);
    out[r] += __shfl_xor_sync(0xffffffffu, out[r], 2);
  }
  return make_float4(out[0], out[1], out[2], out[3]);
}

// MT: n8 tiles of B (four batch rows each, eight with kXV2). GRP: alpha and beta staged per unit and 128-column
// group (always with base-3 codes), else one alpha per row.
template <int MT, int MODE, bool GRP>
__global__ void __launch_bounds__(kXThreads, 1)
    qtea_gemv_mma_kernel(const __grid_constant__ TensorMaps maps, const __grid_constant__ XParams P) {
  constexpr bool BASE3 = MODE <= kXRows, DIAG = MODE == kXDiag, VENC = MODE == kXV2;
  constexpr int NV = VENC ? 4 : 2;  // values of a thread per row block and tile
  // 2-bit codes with v*x split: a unit's sum, residual included, is formed on its own before it joins the tile's, one
  // rounding beside the tile's sum for 512 columns (Qwen3-14B layer, M = 4: errors of 0.80e-7 against 0.90e-7 of the
  // outputs' norm and 32.8 against 32.4 us, with the accumulators folded twice a unit; the kernel before: 0.82e-7)
  constexpr bool kUnit = MODE == kXSplit2;
  // SETS sets of H helper warps take units in turn; CW consumer warps of BLK 16-row blocks
  constexpr int H = kXHelpers, SETS = kXSets, BLK = kXBlocks, CW = kXTileRows / 16 / BLK;
  constexpr int kXHelperThreads = 32 * H;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  uint8_t* smem = smem_raw + (BASE3 ? 0u : (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int u0 = cta_unit_begin(blockIdx.x, P.unit_q, P.unit_r, gridDim.x);
  const int u1 = cta_unit_begin(blockIdx.x + 1, P.unit_q, P.unit_r, gridDim.x), n_units = u1 - u0;
  const int S = P.n_stages, row_slot = P.row_slot, NP = P.n_problems, M = P.M;
  const XStage lay = x_stage_layout(MODE, MT, row_slot);
  XProblem* tab = reinterpret_cast<XProblem*>(smem + (size_t)S * lay.total);
  uint64_t* full = reinterpret_cast<uint64_t*>(tab + kMaxProblems);  // [S] the helpers' copies and stores landed
  uint64_t* empty = full + S;                                        // [S] consumers released it
  uint32_t* boff = reinterpret_cast<uint32_t*>(empty + S);           // [64] x_b_offset of two columns each
  {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(P.prob);
    uint32_t* dst = reinterpret_cast<uint32_t*>(tab);
    for (int i = threadIdx.x; i < NP * (int)(sizeof(XProblem) / 4); i += kXThreads) dst[i] = src[i];
  }
  uint2* mask = reinterpret_cast<uint2*>(boff + 64);                 // [256] x_mask
  // batch rows with products left out of B, by chunk (chunk % kXOutWords: bits that a chunk does not need do no harm),
  // then over all chunks
  uint32_t* left_out = reinterpret_cast<uint32_t*>(mask + 256);
  for (int i = threadIdx.x; i <= kXOutWords; i += kXThreads) left_out[i] = 0u;
  for (int i = threadIdx.x; i < 256; i += kXThreads) mask[i] = x_mask((uint32_t)i);
  if (BASE3 && threadIdx.x < 64)
    boff[threadIdx.x] = x_b_offset<DIAG>(2 * threadIdx.x) | x_b_offset<DIAG>(2 * threadIdx.x + 1) << 16;
  // B columns that no batch row (or, with DIAG, no lane's block) writes, and k slots of pad digits, stay
  // zero in every stage; the scales of rows past N too
  for (int s = 0; s < S; ++s) {
    uint4* z = reinterpret_cast<uint4*>(smem + (size_t)s * lay.total + lay.scales);
    for (int i = threadIdx.x; i < (lay.b_end - lay.scales) / 16; i += kXThreads) z[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(smem_u32(&full[i]), 2 * kXHelperThreads + (P.tma ? 1 : 0));  // a thread's copies, its stores; the TMA
      mbar_init(smem_u32(&empty[i]), CW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp < SETS * H) {
    // ---------------------------------------------------------------- helpers
    const int set = warp / H, hw = warp - set * H, ht = threadIdx.x - set * kXHelperThreads;
    const uint64_t pol = l2_evict_first_policy();
    auto advance = [&](XPos& d) {
#pragma unroll
      for (int k = 0; k < SETS; ++k) x_next(d, tab[d.p], tab[d.p]);
    };
    XPos c = x_pos(tab, NP, u0);
    for (int k = 0; k < set; ++k) x_next(c, tab[c.p], tab[c.p]);
    // a unit's codes: one TMA box where rows are whole 16-byte vectors, else copies by every helper thread
    const bool tma = P.tma != 0;
    auto issue_codes = [&](const XPos& d, int st) {
      uint8_t* sb = smem + (size_t)st * lay.total;
      if (BASE3 && !tma) {
        x_issue_codes<H>(tab[d.p], d, smem_u32(sb), row_slot, ht);
      } else if (ht == 0) {
        const uint32_t bar = smem_u32(&full[st]);
        mbar_arrive_expect_tx(bar, kXTileRows * (BASE3 ? kXBoxBytes : kChunkRowBytes));
        tma_load_2d_hint(smem_u32(sb), &maps.m[d.p], BASE3 ? (d.ch * kXChunkBytes) & ~15 : d.ch * kChunkRowBytes,
                         d.t * kXTileRows, bar, pol);
      }
    };
    {
      // the codes belong to the library and no kernel writes them: the first stages' copies start
      // before the grid dependency wait
      XPos f = c;
      for (int i = set; i < S && i < n_units; i += SETS) {
        issue_codes(f, i);
        advance(f);
      }
    }
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // a unit's loads to registers go out a unit ahead: x of the warp's R batch rows and v, the
    // positions, the salient columns (x there at the unit's start)
    constexpr int R = DIAG ? 1 : (VENC ? 8 : 4) * MT / H;
    XRows<R> rows;
    XPosBytes pos;
    int col = 0, col_next = 0;  // the lane's salient column of c, of n1
    XPos n1 = c;  // the set's unit after c
    auto load_ahead = [&](const XPos& d) {
      const XProblem& a = tab[d.p];
      const int rsn = x_res_steps(d, a);
      x_load_rows<R>(a, d.ch, hw, H, M, VENC ? hw == 0 : hw < M, lane, rows);
      x_load_pos(a, d, d.rs, rsn, ht, pos);
    };
    auto load_sal = [&](const XPos& d) {
      const XProblem& a = tab[d.p];
      return x_has_sal(a, d.rs, x_res_steps(d, a), lane) ? __ldg(a.sal + 16 * d.rs + lane) : 0;
    };
    if (set < n_units) {
      col = load_sal(c);
      load_ahead(c);
    }
    for (int i = set; i < n_units; i += SETS) {
      const int st = i % S;
      uint8_t* sb = smem + (size_t)st * lay.total;
      const XProblem& a = tab[c.p];
      const int rsn = x_res_steps(c, a);
      const bool has_sal = x_has_sal(a, c.rs, rsn, lane);
      if (i + SETS < n_units) {
        advance(n1);
        col_next = load_sal(n1);
      }
      if (i >= S) {
        if (!mbar_wait(smem_u32(&empty[st]), (uint32_t)((i / S - 1) & 1), P.status)) break;
        issue_codes(c, st);
      }
      uint16_t xs[R];
#pragma unroll
      for (int k = 0; k < R; ++k) xs[k] = hw + k * H < M && has_sal ? x_at_sal(a, hw + k * H, col) : (uint16_t)0;
      if (GRP) x_stage_scales<H>(a, c, sb + lay.scales, ht);
      if (rsn > 0) {
        x_stage_residual(a, c, c.rs, rsn, sb + lay.rvals, ht);
        if (ht < kXTileRows / 2)
          *reinterpret_cast<uint32_t*>(sb + lay.rpos + 4 * ht) = pos.b[0] | pos.b[1] << 8 | pos.b[2] << 16 | pos.b[3] << 24;
      }
      x_cp_arrive(smem_u32(&full[st]));
      const int half = (min(32, (a.K - c.ch * kXChunkCols + 15) / 16) + 1) / 2;
      uint32_t maybe = 0u;  // bit m: batch row m may need another E; bit 16 + m: some x at a salient column is not finite
#pragma unroll
      for (int k = 0; k < R; ++k) {
        const int m = hw + k * H;
        if (m >= M) break;
        if (!VENC && rsn > 0) {
          if (!x_finite(xs[k])) {
            maybe |= 0x10000u << m;
            xs[k] = 0;
          }
        }
        const int tile = VENC ? m >> 3 : m >> 2, n = VENC ? m & 7 : 2 * (m & 3);
        if (lane < 16 * rsn)  // x at the salient entries: the row's column, or the hi column of its pair
          *reinterpret_cast<uint16_t*>(sb + lay.rb + tile * kXResBBytes +
                                       ((lane >> 4) * 32 + 4 * n + ((lane >> 2) & 3)) * 8 + 2 * (lane & 3)) = xs[k];
        float* fold = reinterpret_cast<float*>(sb + lay.fold);
        float* sx = reinterpret_cast<float*>(sb + lay.sx);
        bool look;
        if constexpr (BASE3) look = x_build_row<DIAG>(rows.x[k], rows.v, m, boff, sb + lay.b, fold, sx, half, lane);
        else look = x_build_row2<!VENC, GRP>(rows.x[k], rows.v, m, sb + lay.b, fold, sx, half, lane);
        if (look) maybe |= 1u << m;
        if (VENC && m == 0) x_build_v(rows.v, sb + lay.v, lane);
      }
      if constexpr (!VENC) {
        maybe = __reduce_or_sync(0xffffffffu, maybe);
        if (maybe) {
          uint32_t rows_out = maybe >> 16;
          for (uint32_t rest = maybe & 0xFFFFu; rest; rest &= rest - 1u) {
            const int m = __ffs((int)rest) - 1;
            if (x_search<BASE3, DIAG>(a, c.ch, m, reinterpret_cast<float*>(sb + lay.fold), boff, sb + lay.b))
              rows_out |= 1u << m;
          }
          if (rows_out && lane == 0) {
            atomicOr(left_out + (c.ch & (kXOutWords - 1)), rows_out);
            atomicOr(left_out + kXOutWords, rows_out);
          }
        }
      }
      mbar_arrive(smem_u32(&full[st]));
      c = n1;
      col = col_next;
      if (i + SETS < n_units) load_ahead(c);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");  // no copy in flight when the CTA exits
    if (tma && ht == 0)
      for (int j = n_units < S ? 0 : n_units - S; j < n_units; ++j)
        if (j % SETS == set && !mbar_wait(smem_u32(&full[j % S]), (uint32_t)((j / S) & 1), P.status)) break;
    return;
  }

  // ---------------------------------------------------------------- consumers
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int g = lane >> 2, q = lane & 3, tr = (warp - SETS * H) * 16 * BLK;
  const int ct = threadIdx.x - SETS * kXHelperThreads;
  // [row block][tile][value]: rows g and g + 8 of batch row 4 tile + q (DIAG: block q's share); VENC: (row, batch
  // row 8 tile + 2q + 0 / 1)
  float run[BLK][MT][NV];
  auto clear = [&] {
#pragma unroll
    for (int k = 0; k < BLK; ++k)
#pragma unroll
      for (int j = 0; j < MT; ++j)
#pragma unroll
        for (int z = 0; z < NV; ++z) run[k][j][z] = 0.f;
  };
  clear();
  float al[2 * BLK];  // the rows' alpha (without GRP), loaded with a tile's first unit
  bool need_alpha = true;
  int st = 0;
  uint32_t par = 0;
  XPos c = x_pos(tab, NP, u0);
  XShape cur = x_shape(tab[c.p]);
  for (int u = u0; u < u1; ++u) {
    const uint8_t* sb = smem + (size_t)st * lay.total;
    const XProblem& a = tab[c.p];
    if (!GRP && need_alpha) {
#pragma unroll
      for (int r = 0; r < 2 * BLK; ++r) {
        const int row = c.t * kXTileRows + tr + 8 * r + g;
        al[r] = row < a.N ? h2f(__ldg(a.scales + row)) : 0.f;
      }
      need_alpha = false;
    }
    if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&full[st]), par, P.status))) break;
    const uint8_t* sc = sb + lay.scales + (tr + g) * 16;
    const float* fold = reinterpret_cast<const float*>(sb + lay.fold);
    const float* sx = reinterpret_cast<const float*>(sb + lay.sx);
    // base-3 rows start at their own offset in their slots
    const int off = BASE3 ? (int)(((size_t)(tr + g) * a.row_bytes + (size_t)c.ch * kXChunkBytes) & 15) : 0;
    const uint8_t* row = sb + (tr + g) * row_slot;
    const int rsn = x_res_steps(c, cur);
    float unit[BLK][MT][NV];
    if constexpr (kUnit) {
#pragma unroll
      for (int k = 0; k < BLK; ++k)
#pragma unroll
        for (int j = 0; j < MT; ++j)
#pragma unroll
          for (int z = 0; z < NV; ++z) unit[k][j][z] = 0.f;
    }
    float (&sums)[BLK][MT][NV] = kUnit ? unit : run;
    if constexpr (!BASE3) {
      x_decode2<MT, BLK, !VENC, GRP>(sb + (tr + g) * kChunkRowBytes + 4 * q, sb + lay.b, sb + lay.v, sc, fold, sx,
                                     a.bias != 0, al, g, q, lane, P, sums);
    } else if constexpr (DIAG) {
      // the lane's block: 2^-E, alpha, and beta times its sum of x
      const int o0 = off + 26 * q;
      float sum[BLK][2];
      x_decode_diag<BLK>(row + (o0 & ~3), row_slot, 8 * (o0 & 2), sb + lay.b, lane, sum);
      const float F = fold[0], bx = a.bias ? sx[16 * q] : 0.f;
#pragma unroll
      for (int r = 0; r < 2 * BLK; ++r) {
        const uint32_t ab = *reinterpret_cast<const uint32_t*>(sc + r * 128 + 4 * q);
        run[r >> 1][0][r & 1] += fmaf(h2f((uint16_t)ab), sum[r >> 1][r & 1] * F, h2f((uint16_t)(ab >> 16)) * bx);
      }
    } else {
      bool tiny = false;
      x_decode_rows<MT, BLK>(row, off, row_slot, sb + lay.b, sc, fold, sx, a.bias != 0, q, lane, tiny, run);
      if (tiny) {
        atomicOr(left_out + (c.ch & (kXOutWords - 1)), (1u << M) - 1u);
        atomicOr(left_out + kXOutWords, 1u);
      }
    }
    if (rsn > 0) {
      float acc[BLK][MT][4];
#pragma unroll
      for (int k = 0; k < BLK; ++k)
#pragma unroll
        for (int j = 0; j < MT; ++j)
#pragma unroll
          for (int z = 0; z < 4; ++z) acc[k][j][z] = 0.f;
      for (int s = 0; s < rsn; ++s)
        x_res_step<MT, BLK>(sb + lay.rvals, sb + lay.rpos, sb + lay.rb, mask, s, a.fp8 != 0, tr, g, q, lane, acc);
#pragma unroll
      for (int k = 0; k < BLK; ++k)
#pragma unroll
        for (int j = 0; j < MT; ++j)
#pragma unroll
          for (int z = 0; z < NV; ++z) sums[k][j][z] += acc[k][j][VENC ? z : 2 * z];
    }
    if constexpr (kUnit) {
#pragma unroll
      for (int k = 0; k < BLK; ++k)
#pragma unroll
        for (int j = 0; j < MT; ++j)
#pragma unroll
          for (int z = 0; z < NV; ++z) run[k][j][z] += unit[k][j][z];
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(smem_u32(&empty[st]));

    if (c.ch == cur.n_chunks - 1 || u == u1 - 1) {
      // ---- the tile's epilogue once this CTA's part of it is done
      const int A = a.unit_begin + c.t * a.n_chunks, B = A + a.n_chunks;
      if constexpr (VENC) {
        uint32_t again = 0u;  // batch rows with a sum that is not finite
#pragma unroll
        for (int j = 0; j < MT; ++j)
#pragma unroll
          for (int z = 0; z < 2; ++z) {
            float f = 0.f;
#pragma unroll
            for (int r = 0; r < 2 * BLK; ++r) f = fmaf(run[r >> 1][j][2 * (r & 1) + z], 0.f, f);
            if (f != 0.f) again |= 1u << (8 * j + 2 * q + z);
          }
        again = __reduce_or_sync(0xffffffffu, again) & ((1u << M) - 1u);
        for (; again; again &= again - 1u) {
          const int m = __ffs((int)again) - 1;
          const float4 s4 = x_again(a, max(u0 - A, 0), c.ch, m, c.t * kXTileRows + tr + g);
          const float sum[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
          for (int j = 0; j < MT; ++j)
#pragma unroll
            for (int z = 0; z < 2; ++z)
              if (8 * j + 2 * q + z == m)
#pragma unroll
                for (int r = 0; r < 2 * BLK; ++r) run[r >> 1][j][2 * (r & 1) + z] = sum[r];
        }
      } else if (__any_sync(0xffffffffu, left_out[kXOutWords] != 0u)) {
        for (int ch = max(u0 - A, 0); ch <= c.ch; ++ch) {
          // read once for the warp: the helpers may be adding bits for later units
          uint32_t rows_out = __shfl_sync(0xffffffffu, left_out[ch & (kXOutWords - 1)], 0);
          for (; rows_out; rows_out &= rows_out - 1u) {
            const int m = __ffs((int)rows_out) - 1;
            const float4 o4 = x_left_out<BASE3, DIAG>(a, ch, m, c.t * kXTileRows + tr + g);
            const float add[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
            for (int j = 0; j < MT; ++j)
#pragma unroll
              for (int r = 0; r < 2 * BLK; ++r) run[r >> 1][j][r & 1] += 4 * j + q == m ? add[r] : 0.f;
          }
        }
      }
      if (DIAG) {  // the four blocks' shares, in lane order
#pragma unroll
        for (int k = 0; k < BLK; ++k)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            run[k][0][h] += __shfl_xor_sync(0xffffffffu, run[k][0][h], 1);
            run[k][0][h] += __shfl_xor_sync(0xffffffffu, run[k][0][h], 2);
          }
      }
      constexpr int kWords = BLK * MT * NV;
      bool write = true;
      if (A < u0) {
        // not the first contributor: this CTA's partial rows, word by word (slot of this CTA)
        uint32_t* mine = a.part + (size_t)blockIdx.x * kWords * (32 * CW) + ct;
        if (!DIAG || q == 0) {
#pragma unroll
          for (int z = 0; z < kWords; ++z)
            x_part_store(mine + z * (32 * CW), __float_as_uint(run[z / (MT * NV)][z / NV % MT][z % NV]) ^ kXPartEmpty);
        }
        write = false;
      } else if (B > u1) {
        // first contributor of a split tile: the partners' partial rows in CTA order, emptied again
        const int last = x_unit_owner(B - 1, P.total_units, gridDim.x);
        bool timed_out = false;
        for (int cb = (int)blockIdx.x + 1; cb <= last; ++cb) {
          uint32_t* src = a.part + (size_t)cb * kWords * (32 * CW) + ct;
          if (!DIAG || q == 0) {
            uint32_t w[kWords];
#pragma unroll
            for (int z = 0; z < kWords; ++z) w[z] = x_part_load(src + z * (32 * CW));
#pragma unroll
            for (int z = 0; z < kWords; ++z) {
              if (!timed_out && w[z] == 0u) {
                const unsigned long long t0 = global_ns();
                do {
                  w[z] = x_part_load(src + z * (32 * CW));
                  if (global_ns() - t0 > kWaitLimitNs) {
                    atomicExch(P.status, (int)QTEA_ERR_TIMEOUT);
                    timed_out = true;
                    break;
                  }
                } while (w[z] == 0u);
              }
              run[z / (MT * NV)][z / NV % MT][z % NV] += __uint_as_float(w[z] ^ kXPartEmpty);
              x_part_store(src + z * (32 * CW), 0u);
            }
          }
        }
      }
      if (write) {
#pragma unroll
        for (int k = 0; k < BLK; ++k)
#pragma unroll
          for (int z = 0; z < NV; ++z) {
            const int row = c.t * kXTileRows + tr + 16 * k + 8 * (VENC ? z >> 1 : z) + g;
#pragma unroll
            for (int j = 0; j < MT; ++j) {
              const int m = DIAG ? 0 : VENC ? 8 * j + 2 * q + (z & 1) : 4 * j + q;
              if (row < a.N && m < M && (!DIAG || q == 0)) a.y[(size_t)m * a.N + row] = run[k][j][z];
            }
          }
      }
      clear();
      need_alpha = true;
    }
    if (++st == S) {
      st = 0;
      par ^= 1u;
    }
    if (x_next(c, cur, a) && u + 1 < u1) cur = x_shape(tab[c.p]);
  }
}

template <int MT, int MODE, bool GRP>
cudaError_t x_configure(size_t smem_optin) {
  return cudaFuncSetAttribute(qtea_gemv_mma_kernel<MT, MODE, GRP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)smem_optin);
}
template <int MT, int MODE, bool GRP>
cudaError_t x_launch(const TensorMaps& maps, const XParams& p, int grid, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)kXThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, qtea_gemv_mma_kernel<MT, MODE, GRP>, maps, p);
}

}  // namespace
}  // namespace qtea
