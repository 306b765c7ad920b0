// The integer-grid split of the float32 path's tensor-core sweeps.
//
// tcgen05 products accumulate with truncation: every K = 16 step cuts the running sum
// toward zero at its 24th bit (measured on GB300: a chain of 4 steps is 0.58 ulp low on
// average, 64 steps 7 ulp), where a float32 FMA chain rounds to nearest and is unbiased. A
// bias common to a row goes straight into its log-sum-exp, so a plain hi/lo split is not
// good enough for the float32 path. Here the leading part of every operand is an integer:
// with v = sqrt(c) (x - mu) 2^e and e chosen per cloud so that the largest row norm lies
// in [2^10, 2^11),
//   v = h + l + r,  h = rint(v) (|h| <= 2048: exact in half precision),
//   l = half(v - h), r = half(v - h - l)  (what is left is below 2^-24),
// so that every partial sum of h . h' is an integer below 2^22 and accumulates without any
// rounding. The other products (h l', l h', l l', h r', r h': 2^-11 of the first and less)
// go to a second accumulator, whose own truncation is 2^-24 of that, and so do l r' and r l'
// where far points leave the ordinary ones a small part of the grid (grid_reach); the bias is split
// into its integer part (first accumulator, exact) and its fraction (second). The LSE
// warps add the two accumulators with one rounding to nearest. So t_ij carries half an
// ulp, less than the float32 chain of any d, and nothing depends on the order of the
// products.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "progot_common.cuh"
#include "tc_common.cuh"

namespace progot {

// Exponents of the two clouds from their largest squared row norms and sqrt(c): the
// scaled norms lie in [2^10, 2^11); never above 2^9 and 2^10 (clouds that are small
// against eps), so that the scaled bias, whose log2 weight alone is about log2 n, keeps
// its integer part below 2^24.
__device__ __forceinline__ int grid_exp(float norm2_max, float sc, int cap) {
  const float a = sqrtf(norm2_max) * sc;
  if (!(a > 0.f) || !isfinite(a)) return 0;
  int k;
  frexpf(a, &k);  // a < 2^k
  return max(-60, min(cap, 11 - k));
}
struct GridScale {
  int ex, ey;
  float s2;   // 2^(ex + ey)
  float inv;  // 2^-(ex + ey)
};
// hull: the x cloud moved inside the hull of both since its norms were taken; the larger of
// both clouds' norms bounds every point of it.
__device__ __forceinline__ GridScale grid_scale(const GridWords& w, float sc, bool hull) {
  GridScale g;
  const float a = w.norm2_max[0], b = w.norm2_max[1];
  g.ex = grid_exp(hull ? __int_as_float(max(__float_as_int(a), __float_as_int(b))) : a, sc, 9);
  g.ey = grid_exp(b, sc, 10);
  g.s2 = ldexpf(1.f, g.ex + g.ey);
  g.inv = ldexpf(1.f, -(g.ex + g.ey));
  return g;
}

// What the split loses on these clouds beside the CUDA cores' float32 chain, which carries a pair
// of ordinary points to 2^-24 |x||y| c (uncentred; norms of ordinary points are geometric means, to
// powers of two). A point's parts resolve 2^-25 units, 2^-36 of its cloud's largest norm, so the
// grid has t to 2^-36 max|x~| |y~| c, and the same with the sides swapped: when far points set the
// grid (or pull the centre away) by more than 2^10 (d <= 64), x2 below, the CUDA cores are the more exact and
// the clouds are left to them. Without the products l r' and r l' (2^-14 units a coordinate) it has
// 2^-39 sqrt(d) max|x~| max|y~| c: they are formed beyond 2^8, x1 below, where that reaches the
// chain's. (300 x 300, d = 64, one point of each cloud moved out by k spreads, relative error of
// the other rows' sums: k = 100 2.8e-6 without them and 3e-7 with, k = 300 2.4e-5 and 3e-7, the
// chain 3e-7.) With many coordinates an ordinary point beside a far one has its leading parts near
// zero, so that the second accumulator carries the sums and truncates them at every K step: 1.2 bits
// of reach for every doubling of d beyond 64 (a map beside one far y, rms error of the others against
// the CUDA cores': d = 300, 64 spreads 6.0e-8 against 7.5e-8 and 300 spreads 2.1e-7; d = 1000, 32
// spreads 4.7e-8 against 4.4e-8 and 64 spreads 1.1e-7; d = 3000, 16 spreads 5.1e-8 against 4.3e-8
// and 64 spreads 2.3e-7), at most 7.5, so that clouds without far points stay. Below ex + ey = 0 t exceeds 2^22 and float32 log-sum-exps of it lose whole units;
// a norm that is not finite has no grid at all: both are left to the CUDA cores too.
struct GridReach {
  float x1, x2;  // log2
};
__device__ __forceinline__ GridReach grid_reach(const GridWords& w, int d, bool hull) {
  const float a = w.norm2_max[0], b = w.norm2_max[1];
  GridReach r = {0.f, 0.f};
  if (w.nonzero[0] == 0u || w.nonzero[1] == 0u || !(a > 0.f) || !(b > 0.f)) return r;
  // log2 of: largest norms, ordinary norms about the centre and about the origin
  float ax = 0.5f * (float)ilogbf(a);
  const float ay = 0.5f * (float)ilogbf(b);
  float cx = (float)(0.5 * (double)w.exp_sum[0] / (double)w.nonzero[0]);
  const float cy = (float)(0.5 * (double)w.exp_sum[1] / (double)w.nonzero[1]);
  float rx = (float)(0.5 * (double)w.raw_sum[0] / (double)w.nonzero[0]);
  const float ry = (float)(0.5 * (double)w.raw_sum[1] / (double)w.nonzero[1]);
  if (hull) {
    ax = fmaxf(ax, ay);
    cx = fmaxf(cx, cy);
    rx = fminf(rx, ry);
  }
  r.x1 = ax + ay - (rx + ry) + fmaxf(0.f, 0.5f * log2f((float)d) - 3.f);
  r.x2 = fmaxf(ax + cy, ay + cx) - (rx + ry) + fminf(7.5f, 1.2f * fmaxf(0.f, log2f((float)d) - 6.f));
  return r;
}
constexpr float kGridCross = 8.f, kGridReach = 10.f;
__device__ __forceinline__ bool grid_out_of_range(const GridWords& w, const GridScale& g, const GridReach& r,
                                                  int min_exp) {
  return !isfinite(w.norm2_max[0]) || !isfinite(w.norm2_max[1]) || g.ex + g.ey < min_exp || r.x2 > kGridReach;
}

// beta = (pot - norm) bscale as an unevaluated sum of two floats (hi + lo): a float32 beta
// would carry half an ulp of its own, and the rounding of bscale against sqrt(c) a relative
// error common to all pairs.
__device__ __forceinline__ float2 grid_beta(float pot, float norm, float bscale, float bscale_lo) {
  const float d = pot - norm;
  const float bb = d - pot;
  const float de = (pot - (d - bb)) - (norm + bb);
  const float h = d * bscale;
  if (!isfinite(h)) return make_float2(h, 0.f);
  return make_float2(h, fmaf(d, bscale, -h) + fmaf(d, bscale_lo, de * bscale));
}

// Below this (units of the accumulators) a score is no score: a padded column's, or one of a point
// masked out by its potential (-inf, zero weight, the type's lowest value). The folds skip a running
// maximum below it, since differences of such values times a sum would overflow.
constexpr float kGridEmpty = -1e30f;

// Bias row (16 bf16 slots) of beta: slots 0-2 the integer part of beta s2 in bf16 pieces
// (added to the first accumulator), slots 8-10 its fraction (second accumulator). What lies
// below kGridEmpty becomes a large negative finite value, since the other accumulator's
// product meets it with a zero; NaN and +inf stay NaN.
__device__ __forceinline__ void write_bias_row_grid(__nv_bfloat16* row16, float2 beta2, float s2) {
  const float bs = beta2.x * s2;
  uint32_t w[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) w[q] = 0u;
  if (bs < kGridEmpty) {
    w[0] = 0xFF7Fu;  // -3.39e38
  } else if (!isfinite(bs)) {
    w[0] = 0x7FC0u;
  } else {
    const float bi = rintf(bs), bf = (bs - bi) + beta2.y * s2;
    const __nv_bfloat16 i1 = __float2bfloat16_rn(bi);
    const float r1 = bi - __bfloat162float(i1);
    const __nv_bfloat16 i2 = __float2bfloat16_rn(r1);
    const __nv_bfloat16 i3 = __float2bfloat16_rn(r1 - __bfloat162float(i2));
    const __nv_bfloat16 f1 = __float2bfloat16_rn(bf);
    const float q1 = bf - __bfloat162float(f1);
    const __nv_bfloat16 f2 = __float2bfloat16_rn(q1);
    const __nv_bfloat16 f3 = __float2bfloat16_rn(q1 - __bfloat162float(f2));
    w[0] = (uint32_t)__bfloat16_as_ushort(i1) | ((uint32_t)__bfloat16_as_ushort(i2) << 16);
    w[1] = (uint32_t)__bfloat16_as_ushort(i3);
    w[4] = (uint32_t)__bfloat16_as_ushort(f1) | ((uint32_t)__bfloat16_as_ushort(f2) << 16);
    w[5] = (uint32_t)__bfloat16_as_ushort(f3);
  }
  uint4* dst = reinterpret_cast<uint4*>(row16);
  dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
  dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

// A sides of the two bias products in 32-byte-swizzled 128-row tiles: ones in slots 0-7
// (first tile) and in slots 8-15 (second tile); chunk c of row r sits at c ^ (r / 4 mod 2).
// ones holds 2 x 4096 bytes; called by nthreads threads of the CTA.
__device__ __forceinline__ void fill_bias_ones_grid(unsigned char* ones, int tid, int nthreads) {
  uint4* dst = reinterpret_cast<uint4*>(ones);
  for (int q = tid; q < 512; q += nthreads) {
    const int tile = q >> 8, row = (q >> 1) & 127, pos = q & 1;
    const int chunk = pos ^ ((row >> 2) & 1);
    const uint32_t v = chunk == tile ? 0x3F803F80u : 0u;
    dst[q] = make_uint4(v, v, v, v);
  }
}

namespace tc {

// The products of one B part of a K block (part 0: h', 1: l', 2: r') with the A parts that
// meet it, KS steps of K = 16: only h h' goes to the first accumulator d1. Unrolled, so
// that the descriptors are constants apart from their base (at N = 128 a product lasts 64
// cycles, about what a loop around it costs the issuing thread).
template <int BN, int KS>
__device__ __forceinline__ void issue_grid_part(int part, uint32_t d1, uint32_t d2, uint64_t ah, uint64_t al,
                                                uint64_t ar, uint64_t bp, uint32_t more) {
  constexpr uint32_t kId = make_idesc_f16(BM, BN);
  if (part == 0) {
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
      // +32 bytes per K = 16 step inside the 128-byte swizzle atom (encoded >> 4)
      umma_id(d1, ah + kk * 2, bp + kk * 2, kId, kk > 0 ? 1u : more);
      umma_id(d2, al + kk * 2, bp + kk * 2, kId, kk > 0 ? 1u : more);
      umma_id(d2, ar + kk * 2, bp + kk * 2, kId, 1u);
    }
  } else if (part == 1) {
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
      umma_id(d2, ah + kk * 2, bp + kk * 2, kId, 1u);
      umma_id(d2, al + kk * 2, bp + kk * 2, kId, 1u);
    }
  } else {
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) umma_id(d2, ah + kk * 2, bp + kk * 2, kId, 1u);
  }
}
// The products r l' and l r' of a K block (GridWords::cross) by the elected lane (on). Out of line:
// in the issue loop their mere presence costs the persistent loop 11 % (1150 us against 1032 for
// 21 updates at 8192^2, d = 64), a call that is not taken nothing.
template <int BN>
__device__ __noinline__ void issue_grid_cross(int ksteps, uint64_t a, uint64_t b, uint32_t d2, bool on) {
  if (!on) return;
  for (int kk = 0; kk < ksteps; ++kk) umma_id(d2, a + kk * 2, b + kk * 2, make_idesc_f16(BM, BN), 1u);
}
template <int BN>
__device__ __forceinline__ void issue_grid_part(int ksteps, int part, uint32_t d1, uint32_t d2, uint64_t ah,
                                                uint64_t al, uint64_t ar, uint64_t bp, uint32_t more) {
  if (ksteps == 4)
    issue_grid_part<BN, 4>(part, d1, d2, ah, al, ar, bp, more);
  else if (ksteps == 3)
    issue_grid_part<BN, 3>(part, d1, d2, ah, al, ar, bp, more);
  else if (ksteps == 2)
    issue_grid_part<BN, 2>(part, d1, d2, ah, al, ar, bp, more);
  else
    issue_grid_part<BN, 1>(part, d1, d2, ah, al, ar, bp, more);
}

}  // namespace tc
}  // namespace progot
