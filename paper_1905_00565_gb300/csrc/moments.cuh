// Skill moments of one query tile in paired FP32 (shared by the search
// kernels; not part of the public ABI).
//
// A tile of kQT queries of one (realization, target) contributes its count, the
// means and centred sums of observed x and predicted y.  x's half is computed
// in FP64 once per (pair, E, tau) (obs_kernel); y's half once per realization,
// which in FP64 is what the epilogue used to wait for: GB300's FP64 pipe takes
// two lanes per SM per clock, five operations a prediction.  Here every
// quantity is an unevaluated sum h + l of two FP32 numbers, built from
// error-free additions and products, so a sum carries about 48 bits; the
// predictions themselves are FP32 values (24 bits).
//
// Values are scaled by a power of two that brings the target series' largest
// magnitude to 2^kScaleBits (exact; rho does not change): squares and their sums
// over a tile stay below 2^112, and there is room below for series whose ordinary
// values are far smaller than their largest.  With c the tile's first prediction
// and b = y - c (exact as h + l), the sums are B1 = sum b, B2 = sum b^2 and AB =
// sum a b, a = x - mean(x) (exact to 48 bits).  y constant over a tile gives
// exactly zero.  From them mean(y) = c + B1/n, Syy = B2 - B1^2/n, Sxy = AB (sum a
// = 0).
//
// A tile whose predictions spread so little against the series' largest value (a
// fill value of 1e30 among values near 1) that its products would leave FP32's
// range at the small end, B2 < kSmallB2, is summed once more in FP64 from the
// predictions themselves, and its record holds three doubles (store_exact).  From
// kSmallB2 on the terms lost below 2^-149 are less than 2^-78 of B2, and, as the
// target's own spread is at least the predictions', less than 2^-70 of sqrt(Sxx
// Syy) in AB.  B2 = 0 means that all predictions are equal, except in a series
// whose values reach below 2^-kDeepBits of its largest: there (SeriesScale)
// such a tile is summed again too.
//
// Order of the sums, the same in every kernel and in both forms: eight
// consecutive queries one after the other, then a binary tree over the tile's 32
// such groups.
#pragma once

#include "ccm_internal.h"

namespace ccm {

constexpr int kQT = 256;                  // queries per tile
constexpr int kMomentGroup = 8;           // queries summed one after the other
constexpr int kVecStride = kQT + 8;       // floats of a staged prediction vector
constexpr unsigned kAllLanes = 0xffffffffu;
constexpr float kSmallB2 = 0x1p-60f;

// Where query q of a tile lies in a staged prediction vector: one pad word per
// 32 queries, so that lanes walking different groups hit different banks.
__device__ __forceinline__ int vec_slot(int q) { return q + (q >> 5); }
// Where query q of a tile lies in a record of centred observations: lanes
// walking the tile's eight runs of 32 queries read consecutive elements.
__device__ __forceinline__ int obs_slot(int q) { return ((q & 31) << 3) | (q >> 5); }

struct Pair32 {
  float h, l;
};

__device__ __forceinline__ float two_sum(float a, float b, float& err) {
  const float s = __fadd_rn(a, b);
  const float v = __fsub_rn(s, a);
  err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, v)), __fsub_rn(b, v));
  return s;
}
__device__ __forceinline__ void accumulate(Pair32& acc, float h, float l) {
  float e;
  acc.h = two_sum(acc.h, h, e);
  acc.l = __fadd_rn(acc.l, __fadd_rn(e, l));
}
// Symmetric in its arguments (both add to the same bits).
__device__ __forceinline__ Pair32 merge_pairs(const Pair32& a, const Pair32& b) {
  Pair32 r;
  float e;
  r.h = two_sum(a.h, b.h, e);
  r.l = __fadd_rn(__fadd_rn(a.l, b.l), e);
  return r;
}

struct TileSums {
  Pair32 b1, b2, ab;
};
__device__ __forceinline__ TileSums zero_sums() {
  TileSums z;
  z.b1 = z.b2 = z.ab = Pair32{0.f, 0.f};
  return z;
}

// One query: y its scaled prediction, a its centred observation {h, l}.
__device__ __forceinline__ void add_query(TileSums& m, float y, float2 a, float c) {
  const float b = __fsub_rn(y, c);  // b + e = y - c exactly
  const float v = __fsub_rn(b, y);
  const float e = __fsub_rn(__fsub_rn(y, __fsub_rn(b, v)), __fadd_rn(c, v));
  accumulate(m.b1, b, e);
  float p = __fmul_rn(b, b);
  float pe = __fmaf_rn(__fadd_rn(b, b), e, __fmaf_rn(b, b, -p));
  accumulate(m.b2, p, pe);
  p = __fmul_rn(a.x, b);
  pe = __fmaf_rn(a.x, e, __fmaf_rn(a.y, b, __fmaf_rn(a.x, b, -p)));
  accumulate(m.ab, p, pe);
}

// Two sums side by side in packed FP32 pairs (one instruction for both halves,
// each rounded as the scalar operation is: the same bits as two add_query).
// Half of the epilogue's instructions are these sums.
using packed = unsigned long long;
__device__ __forceinline__ packed pack2(float lo, float hi) {
  packed r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(packed x, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(x));
}
__device__ __forceinline__ packed add2(packed a, packed b) {
  packed r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ packed sub2(packed a, packed b) {
  packed r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ packed mul2(packed a, packed b) {
  packed r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ packed fma2(packed a, packed b, packed c) {
  packed r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
struct Pair32x2 {
  packed h, l;
};
struct TileSums2 {
  Pair32x2 b1, b2, ab;
};
__device__ __forceinline__ TileSums2 zero_sums2() {
  TileSums2 z;
  z.b1 = z.b2 = z.ab = Pair32x2{0ull, 0ull};
  return z;
}
__device__ __forceinline__ void accumulate2(Pair32x2& acc, packed h, packed l) {
  const packed s = add2(acc.h, h);
  const packed v = sub2(s, acc.h);
  const packed err = add2(sub2(acc.h, sub2(s, v)), sub2(h, v));
  acc.h = s;
  acc.l = add2(acc.l, add2(err, l));
}
// accumulate2 of -n: subtractions in place of a negated operand
__device__ __forceinline__ void accumulate2_negated(Pair32x2& acc, packed n, packed l) {
  const packed s = sub2(acc.h, n);
  const packed v = sub2(s, acc.h);
  const packed err = sub2(sub2(acc.h, sub2(s, v)), add2(n, v));
  acc.h = s;
  acc.l = add2(acc.l, add2(err, l));
}
__device__ __forceinline__ void add_query2(TileSums2& m, packed y, float2 a0, float2 a1, packed c) {
  const packed b = sub2(y, c), nb = sub2(c, y);
  const packed v = sub2(b, y);
  const packed e = sub2(sub2(y, sub2(b, v)), add2(c, v));
  const packed ah = pack2(a0.x, a1.x), al = pack2(a0.y, a1.y);
  accumulate2(m.b1, b, e);
  packed np = mul2(b, nb);
  packed pe = fma2(add2(b, b), e, fma2(b, b, np));
  accumulate2_negated(m.b2, np, pe);
  np = mul2(ah, nb);
  pe = fma2(ah, e, fma2(al, b, fma2(ah, b, np)));
  accumulate2_negated(m.ab, np, pe);
}
__device__ __forceinline__ void unpack_sums(const TileSums2& m, TileSums& lo, TileSums& hi) {
  unpack2(m.b1.h, lo.b1.h, hi.b1.h);
  unpack2(m.b1.l, lo.b1.l, hi.b1.l);
  unpack2(m.b2.h, lo.b2.h, hi.b2.h);
  unpack2(m.b2.l, lo.b2.l, hi.b2.l);
  unpack2(m.ab.h, lo.ab.h, hi.ab.h);
  unpack2(m.ab.l, lo.ab.l, hi.ab.l);
}

__device__ __forceinline__ TileSums merge_sums(const TileSums& a, const TileSums& b) {
  TileSums r;
  r.b1 = merge_pairs(a.b1, b.b1);
  r.b2 = merge_pairs(a.b2, b.b2);
  r.ab = merge_pairs(a.ab, b.ab);
  return r;
}
__device__ __forceinline__ TileSums merge_across(const TileSums& a, int mask) {
  TileSums o;
  o.b1.h = __shfl_xor_sync(kAllLanes, a.b1.h, mask);
  o.b1.l = __shfl_xor_sync(kAllLanes, a.b1.l, mask);
  o.b2.h = __shfl_xor_sync(kAllLanes, a.b2.h, mask);
  o.b2.l = __shfl_xor_sync(kAllLanes, a.b2.l, mask);
  o.ab.h = __shfl_xor_sync(kAllLanes, a.ab.h, mask);
  o.ab.l = __shfl_xor_sync(kAllLanes, a.ab.l, mask);
  return merge_sums(a, o);
}
__device__ __forceinline__ void store_sums(float4* part, float c, const TileSums& m) {
  part[0] = make_float4(c, m.b1.h, m.b1.l, m.b2.h);
  part[1] = make_float4(m.b2.l, m.ab.h, m.ab.l, 0.f);
}

__device__ __forceinline__ bool too_small(float b2, const SeriesScale& s) {
  return b2 < kSmallB2 && b2 >= s.least_b2;
}

// A tile's record in FP64 (scaled as the paired sums are): told from paired sums
// by its last word.
__device__ __forceinline__ void store_exact(float4* part, double my, double syy, double sxy) {
  part[0] = make_float4(__int_as_float(__double2loint(my)), __int_as_float(__double2hiint(my)),
                        __int_as_float(__double2loint(syy)), __int_as_float(__double2hiint(syy)));
  part[1] = make_float4(__int_as_float(__double2loint(sxy)), __int_as_float(__double2hiint(sxy)),
                        0.f, 1.f);
}
__device__ __forceinline__ double word_pair(float lo, float hi) {
  return __hiloint2double(__float_as_int(hi), __float_as_int(lo));
}

// Where a tile's observed values lie: x[order[q]], q < nq, with their record.
struct TileTarget {
  const float* x;         // the target series at the manifold's points
  const int32_t* order;   // the tile's queries
  const ObsStat* stat;
  int32_t nq;
};

// The same tile in FP64 by one warp (rare): ys the unscaled predictions (vec_slot
// order).
__device__ __forceinline__ void exact_sums_warp(const TileTarget& t, const float* ys, float4* part) {
  const int q0 = kMomentGroup * (threadIdx.x & 31), q1 = min(q0 + kMomentGroup, t.nq);
  const double scale = t.stat->series.scale, mx = t.stat->mx;
  auto tree = [](double v) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) v = __dadd_rn(v, __shfl_xor_sync(kAllLanes, v, o));
    return v;
  };
  double s = 0.0, syy = 0.0, sxy = 0.0;
  for (int q = q0; q < q1; ++q) s = __dadd_rn(s, __dmul_rn((double)ys[vec_slot(q)], scale));
  const double my = __ddiv_rn(tree(s), (double)t.nq);
  for (int q = q0; q < q1; ++q) {
    const double b = __dsub_rn(__dmul_rn((double)ys[vec_slot(q)], scale), my);
    const double a = __dsub_rn(__dmul_rn((double)t.x[t.order[q]], scale), mx);
    syy = __fma_rn(b, b, syy);
    sxy = __fma_rn(a, b, sxy);
  }
  syy = tree(syy);
  sxy = tree(sxy);
  if ((threadIdx.x & 31) == 0) store_exact(part, my, syy, sxy);
}
// And by one lane, in the same order: y(q) the unscaled prediction of query q.
template <typename Y>
__device__ __forceinline__ void exact_sums_lane(const TileTarget& t, Y y, float4* part) {
  const double scale = t.stat->series.scale, mx = t.stat->mx;
  double my = 0.0, syy = 0.0, sxy = 0.0;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    double lv[3][6];  // pending subtrees: of sum y; of syy and sxy
    double v[3] = {0.0, 0.0, 0.0};
#pragma unroll 1
    for (int g = 0; g < kQT / kMomentGroup; ++g) {
      v[0] = v[1] = v[2] = 0.0;
#pragma unroll 1
      for (int q = kMomentGroup * g; q < min(kMomentGroup * (g + 1), t.nq); ++q) {
        const double ys = __dmul_rn((double)y(q), scale);
        if (pass == 0) {
          v[0] = __dadd_rn(v[0], ys);
        } else {
          const double b = __dsub_rn(ys, my);
          const double a = __dsub_rn(__dmul_rn((double)t.x[t.order[q]], scale), mx);
          v[1] = __fma_rn(b, b, v[1]);
          v[2] = __fma_rn(a, b, v[2]);
        }
      }
      int l = 0;
#pragma unroll 1
      for (int up = g; up & 1; up >>= 1, ++l)
        for (int k = 0; k < 3; ++k) v[k] = __dadd_rn(lv[k][l], v[k]);
      for (int k = 0; k < 3; ++k) lv[k][l] = v[k];
    }
    if (pass == 0) my = __ddiv_rn(v[0], (double)t.nq);
    syy = v[1];
    sxy = v[2];
  }
  store_exact(part, my, syy, sxy);
}

// Moments of one staged vector by one warp: lane g sums queries 8g .. 8g+7,
// then the tree.  ys: the predictions (vec_slot order, queries past nq ignored),
// a: the tile's record (obs_slot order, zero past nq).  True, in every lane: they
// spread too little.
__device__ __forceinline__ bool tile_sums_warp(const float* ys, const float2* a, SeriesScale s, int nq,
                                               float4* part) {
  const int lane = threadIdx.x & 31;
  const float c = __fmul_rn(ys[0], s.scale);
  TileSums m = zero_sums();
#pragma unroll
  for (int i = 0; i < kMomentGroup; ++i) {
    const int q = kMomentGroup * lane + i;
    const float y = __fmul_rn(ys[vec_slot(q)], s.scale);
    add_query(m, q < nq ? y : c, __ldg(a + obs_slot(q)), c);
  }
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) m = merge_across(m, o);
  if (lane == 0) store_sums(part, c, m);
  return too_small(m.b2.h, s);
}

}  // namespace ccm
