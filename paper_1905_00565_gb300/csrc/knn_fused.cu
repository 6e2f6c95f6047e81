// Fused nearest-neighbour search + simplex projection + skill moments.
//
// For one query tile of one realization (paper Sect. 3.2: "finding the E+1
// nearest neighbors for every lagged-coordinate vector", the step the paper
// names as the most time-consuming), every query point of the shadow manifold
// M_j is compared with every library point; the E+1 nearest (itself
// excluded) give the simplex prediction of the target variable (Sect. 2.1),
// and the tile's moments of (observed, predicted) are merged per realization
// into the Pearson skill (Sect. 2.1).
//
// Design (GB300, FP32 on the CUDA cores; E <= 10 is not a dense contraction):
//  * persistent CTAs pull work items, sorted by cost, from an atomic counter;
//    a brute-force item is one to eight query tiles of one realization, so a
//    library that fits one shared-memory tile is staged once for all of them;
//  * each thread owns one query; library points sit in shared memory in
//    pairs, packed {a_e, b_e} per coordinate, so one sub.f32x2 + fma.f32x2
//    pair advances the query's distances to two points;
//  * a broadcast 128-bit load feeds the packed operations directly;
//  * squared distances are accumulated in coordinate order (first term a
//    rounded product, then one fused multiply-add per coordinate), the same
//    rounding sequence the FP32 selection is defined by;
//  * the library is visited in query order from the run nearest each warp's
//    queries (wrapping around); a lane tests one pair of points of the next 32
//    against the box of the warp's queries, and pairs farther than every
//    lane's threshold are never read;
//  * selection: each query keeps the K = E+1 smallest distances seen as a
//    sorted float list in registers (a min/max network, no index
//    bookkeeping), which is its running threshold, and the (squared
//    distance, index) keys of every candidate at or below the threshold in
//    its column of a shared-memory buffer; the column is compacted when it
//    runs full, and at the end a register network sorts what is left, so the
//    E+1 nearest come out in (distance, index) order however the library was
//    visited;
//  * the epilogue forms u_i = exp(-d_i/d_1) (optionally floored), the
//    prediction, and the moments of each (tile, target) in paired FP32
//    (moments.cuh): predictions go to a shared-memory ring whose eight slots
//    are reduced by eight warps at once; a unit of many targets sums them with
//    a lane per target instead (lane_targets); the observed values' half is
//    done once per (j, i, E, tau) by obs_kernel, not once per realization;
//    rho_kernel merges the tiles' moments in a fixed order, so rho does not
//    depend on the schedule.
#include <float.h>
#include <limits.h>
#include <math.h>

#include <initializer_list>

#include "ccm_internal.h"
#include "launch.cuh"
#include "moments.cuh"

namespace ccm {
namespace {

using u64 = unsigned long long;

constexpr int kThreads = 256;             // threads per CTA = queries per tile
static_assert(kQT == kThreads, "one query per thread");
constexpr int kBuf = 22;                  // candidate keys per query (a column of the buffer)
constexpr int kCoordBytes = kTileBytes;   // shared memory for one library tile
constexpr int kChunk = 16;                // a tile is padded to whole chunks of points
constexpr int kBufBytes = kBuf * kThreads * 8;
// Predictions staged for their moments: kRing (tile, target) vectors, reduced
// together, one warp each, when the ring is full.
constexpr int kRing = kThreads / 32;
constexpr int kRingBytes = kRing * kVecStride * 4;
// Scratch of the lane-per-target epilogue: 1 / sum of weights per query, then
// two buffers of the eight warps' sums (six floats a lane).
constexpr int kLaneScratch = kThreads * 4 + 2 * (kThreads / 32) * 6 * 32 * 4;
static_assert(kBuf * kThreads * 8 >= (kMaxE + 1) * kThreads * 8 + kLaneScratch,
              "the lane-per-target epilogue's scratch fits the candidate buffer");
constexpr int kSmemBytes = kCoordBytes + kBufBytes + kRingBytes;
constexpr unsigned kFull = 0xffffffffu;
// Kernel variants picked per E by the autotuner (results are identical):
//   V = 0 "narrow": 4 library points per step, no early termination;
//   V = 1 "wide":   early termination for E >= 3 (after 2 coordinates for
//                   E <= 6, after 3 above), and 8 points per step for E <= 6
//                   (4 above: registers run out).

// Library points per step (two points per packed operand): more points give
// more independent FMA chains per warp.
template <int E, int V>
constexpr int kStepE = (V == 1 && E <= 6) ? 8 : 4;

// Coordinates summed before the early-termination check (E when there is none).
template <int E, int V>
constexpr int kE1 = (V == 1 && E >= 3) ? (E <= 6 ? 2 : 3) : E;

constexpr int kBoxDims = 8;  // coordinates of a warp's query box, at most

template <int E>
struct TileShape {
  static constexpr int EP = E + (E & 1);                        // coordinates padded to even
  static constexpr int D = E < kBoxDims ? E : kBoxDims;         // coordinates the pruning bounds
  // library points per tile: a point pair takes EP*8 bytes of coordinates + 8 of indices
  static constexpr int LT = brute_tile_points(E);
  static_assert(LT >= 64 && LT % 32 == 0, "tile must hold whole warps of chunks");
};

// Squared distances of one query (coordinates duplicated, {q_e, q_e}) to a
// pair of library points whose coordinates are packed {a_e, b_e} starting at
// `c` (16-byte aligned, EP entries): {d2(q, a), d2(q, b)}, accumulated over
// coordinates [EB, EE) onto `acc` in the fixed order (coordinate 0 a rounded
// product, every later one a fused multiply-add).  Calling it for [0, E1)
// and then [E1, E) gives exactly the bits of one call for [0, E).
template <int E, int EB, int EE>
__device__ __forceinline__ u64 sqdist2_range(const u64 (&qc)[E], const u64* c, u64 acc) {
  const ulonglong2* c2 = reinterpret_cast<const ulonglong2*>(c);
#pragma unroll
  for (int e = EB & ~1; e < EE; e += 2) {
    const ulonglong2 v = c2[e / 2];
    if (e >= EB) {
      const u64 d0 = sub2(qc[e], v.x);
      acc = (e == 0) ? mul2(d0, d0) : fma2(d0, d0, acc);
    }
    if (e + 1 < EE && e + 1 >= EB) {
      const u64 d1 = sub2(qc[e + 1], v.y);
      acc = fma2(d1, d1, acc);
    }
  }
  return acc;
}

__device__ __forceinline__ float min3f(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Smallest of N distances (three-input min where possible).
template <int N>
__device__ __forceinline__ float min_all(const float (&d)[N]) {
  float m = d[0];
  int i = 1;
#pragma unroll
  for (; i + 1 < N; i += 2) m = min3f(m, d[i], d[i + 1]);
  if (i < N) m = fminf(m, d[i]);
  return m;
}

// The selection key: (squared distance, manifold index), lexicographic.
__device__ __forceinline__ bool key_less(float d, int l, float kd, int kl) {
  return d < kd || (d == kd && l < kl);
}

// The same key packed in 64 bits: the bits of a non-negative float order
// like its value, so (bits << 32 | index) compares like (d, index).
__device__ __forceinline__ u64 pack_key(float d, int l) {
  return ((u64)__float_as_uint(d) << 32) | (u64)(uint32_t)l;
}
__device__ __forceinline__ float key_dist(u64 k) { return __uint_as_float((uint32_t)(k >> 32)); }
__device__ __forceinline__ int key_index(u64 k) { return (int)(uint32_t)k; }

// A staged (tile, target) prediction vector awaiting its moments.
struct RingMeta {
  const float2* a;    // the tile's centred observations
  float4* part;       // where its sums go
  SeriesScale series;
  int32_t nq;         // valid queries of the tile
  int32_t target, tile;
};

// One of them in FP64 (rare): all it needs follows from the target and the tile.
__device__ __noinline__ void exact_vector(const float* ys, int target, int tile, int nq, float4* part,
                                          const UnitDesc* units, const TargetDesc* targets,
                                          const float* series, const int32_t* order,
                                          const ObsStat* obs_stat) {
  const TargetDesc& tg = targets[target];
  const UnitDesc& u = units[tg.unit];
  exact_sums_warp(TileTarget{series + u.series_off + (int64_t)tg.i * u.n + (u.E - 1) * u.tau,
                             order + u.order_off + (int64_t)tile * kQT, obs_stat + tg.obs_tile + tile, nq},
                  ys, part);
}

// The staged vectors' sums: warps 0..n-1 take one each, in parallel.  Between
// two block barriers: the slots are complete on entry and free again on exit.
__device__ __forceinline__ void flush_ring(const KnnParams& p, const float* ring, const RingMeta* meta,
                                           int n) {
  __syncthreads();
  const int warp = threadIdx.x >> 5;
  if (warp < n) {
    const RingMeta mt = meta[warp];
    const float* ys = ring + warp * kVecStride;
    if (__builtin_expect(tile_sums_warp(ys, mt.a, mt.series, mt.nq, mt.part), 0))
      exact_vector(ys, mt.target, mt.tile, mt.nq, mt.part, p.units, p.targets, p.series, p.order,
                   p.obs_stat);
  }
  __syncthreads();
}

// The epilogue of a unit with many targets (>= kLaneTargets): a lane per
// target.  The weights and neighbours of the tile's queries lie in shared
// memory (keep[s][query], {weight, neighbour}); warp w takes queries 32w ..
// 32w+31 and 32 targets at a time, so a neighbour's values of 32 targets are
// one coalesced read of the time-major series and every lane sums its own
// target's moments in registers, group of eight after group of eight; the
// warps' sums meet in shared memory.  One thread per query and target after
// target instead gathered 4 bytes a lane from as many lines and spent five
// FP64 operations a prediction.  64 variables, N = 5000, r = 25, all pairs:
// brute force and table scan 222 -> 62 ms a run;
// two groups of queries packed 14.4 -> 12.8 of brute force's, byte offsets for
// 64-bit multiply-adds -> 10.6.
// Block-wide; the caller's next use of keep and scratch is behind the closing
// barrier.
template <int E, bool kWide>
__device__ __forceinline__ float lane_prediction(const u64* keep, const float* rus, const char* col,
                                                 int stride, int q) {
  float acc = 0.f;
#pragma unroll
  for (int s = 0; s <= E; ++s) {
    const u64 k = keep[s * kThreads + q];
    const float* at = reinterpret_cast<const float*>(
        col + (kWide ? (int64_t)key_index(k) * stride * 4 : (int64_t)(uint32_t)k));
    acc = __fmaf_rn(key_dist(k), __ldg(at), acc);
  }
  return __fmul_rn(acc, rus[q]);
}

// The targets whose sums this lane stored and whose predictions spread too little
// for them: again in FP64.
template <int E, bool kWide>
__device__ __noinline__ void exact_targets(const u64* keep, const float* rus, const float* st,
                                           int stride, const TargetDesc* tgs, int T, int n_tiles,
                                           int nq, float4* part, const float* x, int64_t n,
                                           const int32_t* order, const ObsStat* stat) {
  for (int t = threadIdx.x; t < T; t += kThreads) {
    float4* to = part + 2 * (int64_t)t * n_tiles;
    if (!too_small(to->w, stat[tgs[t].obs_tile].series)) continue;
    const char* col = reinterpret_cast<const char*>(st + tgs[t].i);
    exact_sums_lane(TileTarget{x + (int64_t)tgs[t].i * n, order, stat + tgs[t].obs_tile, nq},
                    [=](int q) { return lane_prediction<E, kWide>(keep, rus, col, stride, q); }, to);
  }
}

template <int E, bool kWide>
__device__ __forceinline__ void lane_targets(const KnnParams& p, const UnitDesc& u, int tile, int nq,
                                          const u64* keep, const float* rus, float* sums) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int T = u.n_targets, n_tiles = u.n_tiles, stride = u.st_stride;
  const float* st = p.st + u.st_off + (int64_t)(E - 1) * u.tau * stride;
  const TargetDesc* tgs = p.targets + u.tgt_off;
  const float2* obs = p.obs + tgs[0].obs_tile * kQT + (int64_t)tile * kQT * T;
  const int q0 = warp * 32, q1 = min(nq, q0 + 32);
  const int32_t* order = p.order + u.order_off + (int64_t)tile * kQT;
  bool redo = false;
  for (int tc = 0, turn = 0; tc < T; tc += 32, ++turn) {
    const int t = min(tc + lane, T - 1);  // lanes past the last target repeat it
    const TargetDesc& tg = tgs[t];
    const char* col = reinterpret_cast<const char*>(st + tg.i);
    const SeriesScale sc = p.obs_stat[tg.obs_tile + tile].series;
    const float scale = sc.scale;
    auto predict = [&](int q) { return lane_prediction<E, kWide>(keep, rus, col, stride, q); };
    const float c = __fmul_rn(predict(0), scale);
    const float2* a = obs + t;
    // two groups of eight queries side by side (packed), then the next two
    TileSums part[4];
#pragma unroll
    for (int g = 0; g < 4; g += 2) {
      const int qa = q0 + kMomentGroup * g, qb = qa + kMomentGroup;
      if (qb + kMomentGroup <= q1 && p.dbg_xhat == nullptr) {
        const packed cc = pack2(c, c), ss = pack2(scale, scale);
        TileSums2 both = zero_sums2();
#pragma unroll 2
        for (int i = 0; i < kMomentGroup; ++i)
          add_query2(both, mul2(pack2(predict(qa + i), predict(qb + i)), ss),
                     __ldg(a + (int64_t)(qa + i) * T), __ldg(a + (int64_t)(qb + i) * T), cc);
        unpack_sums(both, part[g], part[g + 1]);
      } else {
        for (int h = 0; h < 2; ++h) {
          TileSums one = zero_sums();
          const int qh = qa + kMomentGroup * h;
          for (int q = qh; q < min(qh + kMomentGroup, q1); ++q) {
            const float y = predict(q);
            if (p.dbg_xhat && tc + lane < T) p.dbg_xhat[tg.q_off + order[q]] = y;
            add_query(one, __fmul_rn(y, scale), __ldg(a + (int64_t)q * T), c);
          }
          if (h == 0) part[g] = one;
          else part[g + 1] = one;
        }
      }
      if (g == 0) part[0] = merge_sums(part[0], part[1]);
    }
    part[0] = merge_sums(part[0], merge_sums(part[2], part[3]));
    // [turn & 1][value][warp][lane]
    float* mine = sums + (turn & 1) * (kThreads / 32) * 6 * 32 + warp * 32 + lane;
    const float v[6] = {part[0].b1.h, part[0].b1.l, part[0].b2.h,
                        part[0].b2.l, part[0].ab.h, part[0].ab.l};
#pragma unroll
    for (int x = 0; x < 6; ++x) mine[x * kThreads] = v[x];
    __syncthreads();
    if (warp == (turn & 7) && tc + lane < T) {
      const float* all = sums + (turn & 1) * (kThreads / 32) * 6 * 32 + lane;
      auto load = [&](int w) {
        const float* f = all + w * 32;
        TileSums m;
        m.b1 = Pair32{f[0], f[kThreads]};
        m.b2 = Pair32{f[2 * kThreads], f[3 * kThreads]};
        m.ab = Pair32{f[4 * kThreads], f[5 * kThreads]};
        return m;
      };
      const TileSums lo = merge_sums(merge_sums(load(0), load(1)), merge_sums(load(2), load(3)));
      const TileSums hi = merge_sums(merge_sums(load(4), load(5)), merge_sums(load(6), load(7)));
      const TileSums m = merge_sums(lo, hi);
      store_sums(p.partials + 2 * (u.part_off + (int64_t)t * n_tiles + tile), c, m);
      redo |= too_small(m.b2.h, sc);
    }
  }
  if (__builtin_expect(redo, 0))  // rare, and behind the loop: its registers are the predictions'
    exact_targets<E, kWide>(keep, rus, st, stride, tgs, T, n_tiles, nq,
                            p.partials + 2 * (u.part_off + tile),
                            p.series + u.series_off + (E - 1) * u.tau, u.n, order, p.obs_stat + tile);
  __syncthreads();
}

// Everything after the neighbour search, shared by the brute-force and the
// table paths: dd[0..E] ascending FP32 squared distances (kDist: their
// distances sqrt_hw(d2) already) and nb[0..E] the neighbours of query m
// (itself excluded).  Simplex weights and the
// prediction of every target; each target's prediction vector goes to the
// next ring slot (ring_n, the same in every thread), and a full ring is
// reduced (flush_ring); units of many targets (kLanes: a kernel of their own, so
// that neither epilogue costs the other registers) take lane_targets instead.
// The CTA flushes what is left when it runs out of work.  rho does not depend on which warp reduced which vector, or when.
// `keep` (brute-force path: the thread's own column of the candidate buffer,
// which only this thread uses and which is free once its search is done)
// holds the weights and neighbours in shared memory, so that a reduction
// between two targets finds no live registers to spill; other warps may still
// be searching, so nothing else of the buffer is touched before a barrier.
// kKeep false: they stay in registers (keep: the lane-per-target scratch).
static_assert(kMaxE + 1 <= kBuf, "the epilogue keeps E+1 entries in a candidate column");
template <int E, bool kLanes, bool kKeep, bool kDist = false>
__device__ __forceinline__ void finish_tile(const KnnParams& p, const UnitDesc& u, int tile, int m, bool valid, const float (&dd)[E + 1],
                                            const int (&nb)[E + 1], float* ring, RingMeta* meta,
                                            int& ring_n, u64* keep) {
  const int tid = threadIdx.x;
  const int n_m = u.n_m;
  const int off = (E - 1) * u.tau;
  const int nq = min(kQT, n_m - tile * kQT);  // valid queries of this tile (>= 1)
  // Simplex weights (Sect. 2.1), once per query for every target.  Every
  // floating-point step below is a fixed operation (explicit rounding or a
  // hardware approximation that is the same everywhere), so the brute-force
  // and table kernels, the plain comparator and every batch produce the same
  // bits.
  const float d1 = kDist ? dd[0] : sqrt_hw(dd[0]);
  const float inv_d1 = (d1 > 0.f) ? rcp_hw(d1) : 0.f;
  float w[E + 1];
  int nbc[E + 1];
  float usum = 0.f;
  // simplex_u_dist with the d1 > 0 test taken once: the exponential for every
  // neighbour, replaced by the limit in the rare query whose nearest is at 0
#pragma unroll
  for (int s = 0; s <= E; ++s) w[s] = simplex_exp(kDist ? dd[s] : sqrt_hw(dd[s]), inv_d1);
  if (!(d1 > 0.f)) {
#pragma unroll
    for (int s = 0; s <= E; ++s) w[s] = simplex_limit(kDist ? dd[s] : sqrt_hw(dd[s]));
  }
#pragma unroll
  for (int s = 0; s <= E; ++s) {
    w[s] = fmaxf(w[s], u.wfloor);
    usum = __fadd_rn(usum, w[s]);
    // brute force: an unfilled slot (only possible with non-finite device
    // input) reads, and is reported, in bounds; table entries are in bounds
    nbc[s] = kDist ? nb[s] : min(max(nb[s], 0), n_m - 1);
    if (kKeep) keep[s * kThreads + tid] = ((u64)__float_as_uint(w[s]) << 32) | (uint32_t)nbc[s];
  }
  if constexpr (kLanes) {
    if (!kKeep) {
#pragma unroll
      for (int s = 0; s <= E; ++s)
        keep[s * kThreads + tid] = ((u64)__float_as_uint(w[s]) << 32) | (uint32_t)nbc[s];
    }
    if (p.dbg_nbr && valid)
      for (int t = 0; t < u.n_targets; ++t)
        for (int s = 0; s <= E; ++s)
          p.dbg_nbr[p.targets[u.tgt_off + t].nbr_off + (int64_t)m * (E + 1) + s] =
              key_index(keep[s * kThreads + tid]);
    float* rus = reinterpret_cast<float*>(keep + (E + 1) * kThreads);
    if (kKeep) __syncthreads();  // other warps' columns reach beyond E+1 keys while they search
    rus[tid] = rcp_hw(usum);
    // neighbours as byte offsets into the time-major series while they fit 32 bits
    const uint32_t row_bytes = (uint32_t)u.st_stride * 4u;
    const bool wide = (u64)u.n * row_bytes >> 32 != 0;
    if (!wide) {
#pragma unroll
      for (int s = 0; s <= E; ++s) {
        const u64 k = keep[s * kThreads + tid];
        keep[s * kThreads + tid] = (k & 0xffffffff00000000ull) | ((uint32_t)k * row_bytes);
      }
    }
    __syncthreads();
    if (wide) lane_targets<E, true>(p, u, tile, nq, keep, rus, rus + kThreads);
    else lane_targets<E, false>(p, u, tile, nq, keep, rus, rus + kThreads);
  } else {
    auto weight = [&](int s) {
      return kKeep ? __uint_as_float((uint32_t)(keep[s * kThreads + tid] >> 32)) : w[s];
    };
    auto nbr = [&](int s) { return kKeep ? (int)(uint32_t)keep[s * kThreads + tid] : nbc[s]; };
    for (int t = 0; t < u.n_targets; ++t) {
      const TargetDesc tg = p.targets[u.tgt_off + t];
      const float* si = p.series + u.series_off + (int64_t)tg.i * u.n;
      float acc = 0.f;
#pragma unroll
      for (int s = 0; s <= E; ++s) acc = __fmaf_rn(weight(s), si[nbr(s) + off], acc);
      const float xhat = __fmul_rn(acc, rcp_hw(usum));  // usum >= exp(-1)
      if (valid) {
        if (p.dbg_xhat) p.dbg_xhat[tg.q_off + m] = xhat;
        if (p.dbg_nbr) {
#pragma unroll
          for (int s = 0; s <= E; ++s) p.dbg_nbr[tg.nbr_off + (int64_t)m * (E + 1) + s] = nbr(s);
        }
      }
      const int64_t rec = tg.obs_tile + tile;
      ring[ring_n * kVecStride + vec_slot(tid)] = xhat;
      if (tid == 0)
        meta[ring_n] = RingMeta{p.obs + rec * kQT,
                                p.partials + 2 * (u.part_off + (int64_t)t * u.n_tiles + tile),
                                p.obs_stat[rec].series, nq, (int32_t)(u.tgt_off + t), tile};
      // a full ring is reduced before the next target's vector, or at the end
      if (++ring_n == kRing && t + 1 < u.n_targets) {
        flush_ring(p, ring, meta, kRing);
        ring_n = 0;
      }
    }
    if (ring_n == kRing) {  // the weights and neighbours are dead here
      flush_ring(p, ring, meta, kRing);
      ring_n = 0;
    }
  }
}

// Stage library points [t0, t0 + nt) of a unit's library (query order) into
// shared memory: coordinates in packed pairs, and indices.  The tile is padded
// to whole chunks with sentinel points (NaN coordinates, index INT_MAX): every
// distance to one is NaN, which compares false against any threshold.
// Block-wide; the caller brackets it with barriers.
template <int E>
__device__ __noinline__ void stage_library(const float* sj, const int32_t* lib, int off, int tau,
                                              int t0, int nt, u64* s_coord, int32_t* s_lidx) {
  constexpr int EP = TileShape<E>::EP;
  const int ntp = (nt + kChunk - 1) / kChunk * kChunk;
  for (int a = threadIdx.x; a < ntp; a += kThreads) {
    float* cpair = reinterpret_cast<float*>(s_coord + (size_t)(a >> 1) * EP) + (a & 1);
    const int l = a < nt ? lib[t0 + a] : INT_MAX;
    s_lidx[a] = l;
#pragma unroll
    for (int e = 0; e < E; ++e)
      cpair[2 * e] = a < nt ? sj[l + off - e * tau] : __int_as_float(0x7fffffff);
    if (EP > E) cpair[2 * E] = 0.f;
  }
}

// The library position (in query order) about as far into the library as
// query position pos is into the manifold: floor(L*pos/N_m), in FP32 (only a
// starting point of the scan: any value in [0, L) gives the same result).
__device__ __forceinline__ int library_position(int L, int pos, int n_m) {
  return min(L - 1, __float2int_rz(__fmul_rn((float)L, __fdividef((float)pos, (float)n_m))));
}

// The running threshold: t[0..K) holds the K smallest squared distances (as
// values, ties repeated) of the candidates seen so far, ascending.  Inserting
// x is a min/max network: slot s becomes min(t[s], max(t[s-1], x)), which
// leaves the list unchanged when x is not below t[K-1].
template <int K>
__device__ __forceinline__ void thresh_insert(float (&t)[K], float x) {
#pragma unroll
  for (int s = K - 1; s > 0; --s) t[s] = fminf(t[s], fmaxf(t[s - 1], x));
  t[0] = fminf(t[0], x);
}

// Ascending insertion sort of one thread's candidate column (n keys, stride
// kThreads) in shared memory.
__device__ __forceinline__ void sort_column(u64* col, int n) {
  for (int i = 1; i < n; ++i) {
    const u64 x = col[i * kThreads];
    int j = i - 1;
    for (; j >= 0; --j) {
      const u64 y = col[j * kThreads];
      if (y <= x) break;
      col[(j + 1) * kThreads] = y;
    }
    col[(j + 1) * kThreads] = x;
  }
}

// Batcher's merge exchange for K keys in registers: the pairs it compares, in
// order (Knuth, The Art of Computer Programming 5.2.2, algorithm M).
template <int K>
struct ExchangePairs {
  int a[64], b[64], n;
  constexpr ExchangePairs() : a(), b(), n(0) {
    for (int p = 1; p < K; p *= 2)
      for (int k = p; k >= 1; k /= 2)
        for (int j = k % p; j + k < K; j += 2 * k)
          for (int i = 0; i < k && i + j + k < K; ++i)
            if ((i + j) / (2 * p) == (i + j + k) / (2 * p)) {
              a[n] = i + j;
              b[n++] = i + j + k;
            }
  }
};
template <int K, int I = 0>
__device__ __forceinline__ void sort_keys(u64 (&k)[K]) {
  constexpr ExchangePairs<K> net;
  if constexpr (I < net.n) {
    constexpr int a = net.a[I], b = net.b[I];
    const u64 x = k[a], y = k[b];
    const bool swap = y < x;
    k[a] = swap ? y : x;
    k[b] = swap ? x : y;
    sort_keys<K, I + 1>(k);
  }
}

// Brute-force search of one work item: query tiles [tile0, tile0 + n_chunk)
// of a unit.  When the whole library fits one shared-memory tile
// it is staged once for all of them; each warp starts its scan at the library
// run nearest its own 32 queries (the library is in query order) and wraps
// around.  Larger libraries are staged tile by tile for every query tile.
//
// Selection.  Each query keeps (a) the running threshold t[] of the K = E+1
// smallest squared distances seen (registers, min/max network) and (b) a
// column of the candidate buffer in shared memory with the keys (squared
// distance, index) of every candidate whose distance was at most the threshold
// when it was seen.  Every key that can still be among the final K smallest
// is in the column: a dropped key had a distance above a threshold that is
// itself at least the final K-th smallest value.  The threshold is brought up
// to date warp-wide once some lane has merge_at new candidates (the network is
// cheap: no index bookkeeping); a nearly full column is compacted to the keys
// at or below the threshold, and, if ties still leave it full, sorted and cut
// to the K smallest keys.  At the end the column is compacted and sorted: its
// first K keys are the E+1 nearest neighbours in (distance, index) order,
// exactly the list the sorted insertion of every candidate would give.
template <int E, int V, bool kLanes, bool kStats, bool kPrune>
__device__ void process_item(const KnnParams& p, const UnitDesc& u, int tile0, int n_chunk,
                             unsigned char* smem, RingMeta* meta, float2* qbox, int& ring_n) {
  constexpr int K = E + 1;  // the window keeps m itself out, so E+1 slots suffice
  constexpr int EP = TileShape<E>::EP;
  constexpr int LT = TileShape<E>::LT;
  constexpr int D = TileShape<E>::D;
  const int n_m = u.n_m, L = u.L, tau = u.tau, W = u.theiler;
  const bool single = L <= LT;
  // Shared-memory layout: library indices [LT], coordinates [LT/2][EP] in the
  // first kCoordBytes, then the candidate buffer [kBuf][kThreads].  A library that fits one tile takes only the
  // coordinate rows it needs, and the buffer starts right after them, so its
  // columns reach up to the prediction ring: wider columns need fewer
  // compactions.
  int32_t* s_lidx = reinterpret_cast<int32_t*>(smem);
  u64* s_coord = reinterpret_cast<u64*>(smem + (size_t)LT * 4);
  size_t buf_off = kCoordBytes;
  if (single) {
    const int ntp = (L + kChunk - 1) / kChunk * kChunk;
    buf_off = (size_t)LT * 4 + (size_t)(ntp / 2) * EP * 8;
  }
  u64* s_buf = reinterpret_cast<u64*>(smem + buf_off);
  const int cap = (int)((kCoordBytes + kBufBytes - buf_off) / (kThreads * 8));  // >= kBuf
  float* s_ring = reinterpret_cast<float*>(smem + kCoordBytes + kBufBytes);      // [kRing][kVecStride]

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int off = (E - 1) * tau;
  const float* sj = p.series + u.series_off + (int64_t)u.j * u.n;
  const int32_t* lib = p.lib + u.lib_off;
  const int32_t* order = p.order + u.order_off;
  constexpr int kStep = kStepE<E, V>;
  constexpr int kPairs = kStep / 2;
  const int room = cap - kStep;   // a column above this cannot take another step
  static_assert(K + kStep <= kBuf, "a cut column must leave room for a step");
  const int merge_at = max(1, min(p.merge_at[E], room));
  // the first kInit points of a query's scan go straight into its threshold
  constexpr int kInit = (K + kStep - 1) / kStep * kStep;
  static_assert(kInit <= kChunk && kInit % kStep == 0, "the initial points are whole runs of the first chunk");
  u64* col = s_buf + tid;  // this thread's candidate column

  const int tile1 = min(u.n_tiles, tile0 + n_chunk);
  if (single) {
    __syncthreads();  // the previous item's readers of the tile are done
    stage_library<E>(sj, lib, off, tau, 0, L, s_coord, s_lidx);
    __syncthreads();
  }
  // A warp's 32 queries are consecutive positions of the query order.  For
  // small E (a short search, so the load latency would show) the next tile's
  // query and coordinates are loaded before this tile's epilogue, so their
  // latency overlaps it; for larger E the registers are needed elsewhere.
  constexpr bool kPrefetch = E <= 3;
  int m_nx;
  float c_nx[E];
  auto load_query = [&](int t) {
    const int ps = t * kQT + tid;
    m_nx = order[ps < n_m ? ps : n_m - 1];
#pragma unroll
    for (int e = 0; e < E; ++e) c_nx[e] = sj[m_nx + off - e * tau];
  };
  if (kPrefetch) load_query(tile0);
  for (int tile = tile0; tile < tile1; ++tile) {
    if (!kPrefetch) load_query(tile);
    const int pos = tile * kQT + tid;
    const bool valid = pos < n_m;
    const int m = m_nx;
    u64 qc[E];
#pragma unroll
    for (int e = 0; e < E; ++e) qc[e] = pack2(c_nx[e], c_nx[e]);
    // Bounding box of the warp's queries over the first D coordinates (in shared
    // memory: the registers are the search's).
#pragma unroll
    for (int e = 0; e < D; ++e) {
      float lo = c_nx[e], hi = lo;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(kFull, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(kFull, hi, o));
      }
      if (lane == 0) qbox[warp * kBoxDims + e] = make_float2(lo, hi);
    }
    __syncwarp();
    // the library position nearest this warp's queries (in query order)
    const int aw = library_position(L, tile * kQT + warp * 32, n_m);

    float tl[K];  // running threshold: the K smallest distances so far, ascending
#pragma unroll
    for (int s = 0; s < K; ++s) tl[s] = INFINITY;
    int cnt = 0, done = 0;  // keys in the column; of them, already in tl
    // counting variant only: warp-uniform step counts, per-lane candidates
    uint32_t st_begun = 0, st_full = 0, st_pruned = 0, st_cand = 0, st_slots = 0;

    // bring tl up to date with the column's new keys (lockstep over the lanes)
    auto update = [&]() {
      const int mx = (int)__reduce_max_sync(kFull, (unsigned)(cnt - done));
      if (kStats) {
        st_cand += (uint32_t)(cnt - done);
        st_slots += (uint32_t)mx;
      }
      for (int b = 0; b < mx; ++b) {
        // the distance half of the key; a lane with no new key inserts +inf
        // (a no-op), and a round no lane needs any more is skipped
        const float x = (b < cnt - done)
                            ? reinterpret_cast<const float*>(col + (done + b) * kThreads)[1]
                            : INFINITY;
        if (__any_sync(kFull, x < tl[K - 1])) thresh_insert<K>(tl, x);
      }
      done = cnt;
    };
    // keep the keys at or below the threshold (in order)
    auto compact = [&]() {
      const float th = tl[K - 1];
      const int mx = (int)__reduce_max_sync(kFull, (unsigned)cnt);
      int w = 0;
      for (int b = 0; b < mx; ++b) {
        if (b < cnt) {
          const u64 x = col[b * kThreads];
          if (key_dist(x) <= th) col[(w++) * kThreads] = x;
        }
      }
      cnt = done = w;
    };
    auto make_room = [&]() {
      update();
      if (__any_sync(kFull, cnt > room)) compact();
      if (__any_sync(kFull, cnt > room)) {  // ties at the threshold: keep the K smallest keys
        if (cnt > room) {
          sort_column(col, cnt);
          cnt = done = K;
        }
      }
    };

    // Scan the staged points [0, nt), 32 pairs of points at a time from the
    // pairs around position `base` (a chunk start) on, wrapping around;
    // `first`: the kInit points at `base` fill tl.
    auto scan = [&](int nt, int base, bool first) {
      const int np = (nt + kChunk - 1) / kChunk * (kChunk / 2);
      const int ng = (np + 31) >> 5;
      if (first) {
#pragma unroll
        for (int pp = 0; pp < kInit / 2; ++pp) {
          const int a = base + 2 * pp;
          float d2[2];
          unpack2(sqdist2_range<E, 0, E>(qc, s_coord + (size_t)(a >> 1) * EP, 0ull), d2[0], d2[1]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int l = s_lidx[a + h];
            if (l != INT_MAX && abs(l - m) > W) {
              thresh_insert<K>(tl, d2[h]);
              col[(cnt++) * kThreads] = pack_key(d2[h], l);
            }
          }
        }
        done = cnt;
        if (kStats) {
          st_begun += kInit;
          st_full += kInit;
        }
        if (__any_sync(kFull, cnt > room)) make_room();
      }
      // one aligned run of kPairs pairs from pair `at` on
      auto step = [&](int at) {
        if (kStats) st_begun += kStep;
        // Partial sums over the first E1 coordinates are lower bounds of the
        // full FP32 sums (all terms are >= 0 and rounding is monotone), so a
        // step whose partials are all above every lane's threshold cannot
        // contribute a candidate and skips the remaining coordinates.
        u64 r[kPairs];
#pragma unroll
        for (int pp = 0; pp < kPairs; ++pp)
          r[pp] = sqdist2_range<E, 0, (kE1<E, V>)>(qc, s_coord + (size_t)(at + pp) * EP, 0ull);
        const float th = tl[K - 1];
        float d[kStep];
#pragma unroll
        for (int pp = 0; pp < kPairs; ++pp) unpack2(r[pp], d[2 * pp], d[2 * pp + 1]);
        if (kStats && (kE1<E, V>) == E) st_full += kStep;
        if (!__any_sync(kFull, min_all(d) <= th)) return;
        if constexpr ((kE1<E, V>) < E) {
          if (kStats) st_full += kStep;
#pragma unroll
          for (int pp = 0; pp < kPairs; ++pp) {
            r[pp] = sqdist2_range<E, (kE1<E, V>), E>(qc, s_coord + (size_t)(at + pp) * EP, r[pp]);
            unpack2(r[pp], d[2 * pp], d[2 * pp + 1]);
          }
          if (!__any_sync(kFull, min_all(d) <= th)) return;
        }
        // the run's library indices (one broadcast 16-byte load per four); its pairs
        // that are not kept lie above every threshold, and the first points' runs
        // hold nothing else (both are whole runs)
        int li[kStep];
#pragma unroll
        for (int q4 = 0; q4 < kStep / 4; ++q4) {
          const int4 v = *reinterpret_cast<const int4*>(s_lidx + 2 * at + 4 * q4);
          li[4 * q4] = v.x;
          li[4 * q4 + 1] = v.y;
          li[4 * q4 + 2] = v.z;
          li[4 * q4 + 3] = v.w;
        }
#pragma unroll
        for (int pt = 0; pt < kStep; ++pt) {
          // at or below the threshold (never a sentinel: NaN), outside the
          // exclusion window |l - m| <= W (W = 0 drops only m itself, and
          // the unsigned form tests both sides at once); appended without a
          // branch
          const bool take =
              (d[pt] <= th) & ((unsigned)li[pt] - (unsigned)m + (unsigned)W > 2u * (unsigned)W);
          if (take) col[cnt * kThreads] = pack_key(d[pt], li[pt]);
          cnt += take ? 1 : 0;
        }
        if (__any_sync(kFull, cnt - done >= merge_at || cnt > room)) make_room();
      };
      if constexpr (!kPrune) {
        // nothing to exclude: run after run, without a mask to walk (at E = 1 a run is
        // 20 instructions and the walk 6: N = 20000 in time order, L = 400, r = 100 0.72
        // -> 0.64 ms)
        for (int jg = 0; jg < ng; ++jg) {
          int g = (base >> 6) + jg;
          g -= (g >= ng) ? ng : 0;
          const int end = min(32 * g + 32, np);
#pragma unroll 2
          for (int at = 32 * g; at < end; at += kPairs)
            if (!(first && (unsigned)(at - (base >> 1)) < (unsigned)(kInit / 2))) step(at);
        }
      } else {
#pragma unroll 1
        for (int jg = 0; jg < ng; ++jg) {
          int g = (base >> 6) + jg;
          g -= (g >= ng) ? ng : 0;
          // Pruning, a lane per pair.  gap_e = max(0, lo_e - qhi_e, qlo_e - hi_e)
          // bounds |q_e - x_e| from below for every query q of the warp and both
          // points x of the pair, in FP32 too (rounding is monotone); summed in the
          // distance's own order over the first D coordinates it bounds their FP32
          // squared distances from below.  A pair whose bound exceeds every lane's
          // threshold holds no candidate.
          const float th_max = __uint_as_float(__reduce_max_sync(kFull, __float_as_uint(tl[K - 1])));
          const int pr = 32 * g + lane;
          bool keep = pr < np && !(first && (unsigned)(pr - (base >> 1)) < (unsigned)(kInit / 2));
          if (keep && p.prune) {
            const float2* xp = reinterpret_cast<const float2*>(s_coord + (size_t)pr * EP);
            float lb = 0.f;
#pragma unroll
            for (int e = 0; e < D; ++e) {
              const float2 x = xp[e], qb = qbox[warp * kBoxDims + e];
              const float gp = fmaxf(fmaxf(__fsub_rn(fminf(x.x, x.y), qb.y),
                                           __fsub_rn(qb.x, fmaxf(x.x, x.y))), 0.f);
              lb = (e == 0) ? __fmul_rn(gp, gp) : __fmaf_rn(gp, gp, lb);
            }
            keep = !(lb > th_max);
          }
          unsigned mask = __ballot_sync(kFull, keep);
          if (kStats) st_pruned += 2u * (min(32, np - 32 * g) - __popc(mask)) -
                                   (first && (base >> 6) == g ? (unsigned)kInit : 0u);
          while (mask != 0u) {
            // the next kept pair's aligned run of kPairs: the pairs in reach of a warp's
            // queries lie side by side in the query order, and collecting them one by
            // one was a chain of find-first-bits (short libraries 4.08 -> 3.97 ms, the
            // sweep's brute force 13.3 -> 12.8, N = 10^5 17.2 -> 16.3)
            const int b0 = (__ffs(mask) - 1) & ~(kPairs - 1);
            mask &= ~(((1u << kPairs) - 1u) << b0);
            step(32 * g + b0);
          }
        }
      }
    };

    // The library is staged tile by tile unless it fits one shared-memory tile
    // (staged once per item above); the first library tile visited is the one
    // nearest this query tile (the same order in every warp: the staging is
    // block-wide).
    const int ntiles = single ? 1 : (L + LT - 1) / LT;
    const int first_t = single ? 0 : library_position(L, tile * kQT, n_m) / LT;
    for (int c = 0; c < ntiles; ++c) {
      int ti = first_t + c;
      ti -= (ti >= ntiles) ? ntiles : 0;
      const int t0 = ti * LT, nt = min(LT, L - t0);
      if (!single) {
        __syncthreads();  // the previous library tile has been consumed
        stage_library<E>(sj, lib, off, tau, t0, nt, s_coord, s_lidx);
        __syncthreads();
      }
      const int local = aw - t0;
      const int base = (local >= 0 && local < nt) ? (local / kChunk) * kChunk : 0;
      scan(nt, base, c == 0);
    }
    update();
    compact();
    // the E+1 nearest in (distance, index) order: K keys are left unless some
    // tie with the threshold (or the input is not finite)
    u64 ku[K];
    if (__all_sync(kFull, cnt == K)) {
#pragma unroll
      for (int s = 0; s < K; ++s) ku[s] = col[s * kThreads];
      sort_keys<K>(ku);
    } else {
      sort_column(col, cnt);
#pragma unroll
      for (int s = 0; s < K; ++s) ku[s] = col[s * kThreads];
    }
    if (kStats) {
      const uint32_t cand = __reduce_add_sync(kFull, st_cand);
      const unsigned vq = __popc(__ballot_sync(kFull, valid));
      if (lane == 0) {
        unsigned long long* c = p.stats;
        atomicAdd(&c[kStatPairsBegun], 32ull * st_begun);
        atomicAdd(&c[kStatPairsFull], 32ull * st_full);
        atomicAdd(&c[kStatPairsPruned], 32ull * st_pruned);
        atomicAdd(&c[kStatCandidates], (unsigned long long)cand);
        atomicAdd(&c[kStatMergeSlots], 32ull * st_slots);
        atomicAdd(&c[kStatBruteQueries], (unsigned long long)vq);
        if (tid == 0) atomicAdd(&c[kStatBruteTiles], 1ull);
      }
    }

    // Epilogue: the E+1 nearest (the window kept the query itself out of the
    // list), simplex weights, prediction, moments.
    float dd[E + 1];
    int nb[E + 1];
#pragma unroll
    for (int s = 0; s <= E; ++s) {
      dd[s] = key_dist(ku[s]);
      nb[s] = key_index(ku[s]);
    }
    if (kPrefetch && tile + 1 < tile1) load_query(tile + 1);
    finish_tile<E, kLanes, true>(p, u, tile, m, valid, dd, nb, s_ring, meta, ring_n, s_buf);
  }
}

// --------------------------------------------------------------------------
// Table path of units with several targets whose realizations are not read in
// groups (units with one target, and groups of many: knn_scan.cu): the
// unit's membership bits (by position of the query order) are copied to shared
// memory and each query walks its row of the distance indexing table (sorted
// by (FP32 squared distance, index) over the whole manifold, the query itself
// left out) until it has met E+1 library members outside the exclusion window.
// Those are, in order, the E+1 nearest library neighbours -- the same list the
// brute-force scan produces.  A query whose row holds fewer members scans the
// library.
template <int E>
__device__ __forceinline__ float d2_point(const float* sj, int off, int tau, const float (&q)[E],
                                          int x) {
  float diff = __fsub_rn(q[0], sj[x + off]);
  float acc = __fmul_rn(diff, diff);
#pragma unroll
  for (int e = 1; e < E; ++e) {
    diff = __fsub_rn(q[e], sj[x + off - e * tau]);
    acc = __fmaf_rn(diff, diff, acc);
  }
  return acc;
}

// Shared memory of the table kernel: the epilogue's ring of predictions, the
// walk's records (below), then the membership bits.
//
// A record is one step of the walk (eight consecutive ranks of the row) that
// held members: (step << 8) | flags, flag c marking rank 8*step + c.  A query
// keeps at most E+1 records: [kMaxE+1][kThreads] 16-bit words.
constexpr int kRecBytes = (kMaxE + 1) * kThreads * 2;
static_assert(kWalkMaxR / 8 <= 256, "a record's step index has eight bits");

// One query's walk along its table row (`row`: its entries): records the steps
// with members until it has K of them; returns the members met.
template <int K, typename Index, bool kStats>
__device__ __forceinline__ int table_walk(const Index* row, const int32_t* order, int steps, int m,
                                          int W, const uint32_t* bits, uint16_t* rec, bool active,
                                          uint32_t& st_entries) {
  int got = 0, nrec = 0;
  for (int g = 0; __any_sync(kFull, active && got < K && g < steps); ++g) {
    if (!(active && got < K && g < steps)) continue;
    if (kStats) st_entries += 8u;
    int x[8];  // ranks 8g .. 8g+7
    if (sizeof(Index) == 2) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(row) + g);
      x[0] = v.x & 0xffffu; x[1] = v.x >> 16; x[2] = v.y & 0xffffu; x[3] = v.y >> 16;
      x[4] = v.z & 0xffffu; x[5] = v.z >> 16; x[6] = v.w & 0xffffu; x[7] = v.w >> 16;
    } else {
      const int4 v0 = __ldg(reinterpret_cast<const int4*>(row) + 2 * g);
      const int4 v1 = __ldg(reinterpret_cast<const int4*>(row) + 2 * g + 1);
      x[0] = v0.x; x[1] = v0.y; x[2] = v0.z; x[3] = v0.w;
      x[4] = v1.x; x[5] = v1.y; x[6] = v1.z; x[7] = v1.w;
    }
    uint32_t flags = 0u;
#pragma unroll
    for (int c = 0; c < 8; ++c) flags |= ((bits[x[c] >> 5] >> (x[c] & 31)) & 1u) << c;
    if (W > 0 && flags != 0u) {
      // points inside the exclusion window |l - m| <= W are no neighbours
      // (the row never holds m itself, so W = 0 excludes nothing)
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if ((flags >> c) & 1u) {
          const int l = order[x[c]];
          if ((unsigned)l - (unsigned)m + (unsigned)W <= 2u * (unsigned)W) flags &= ~(1u << c);
        }
    }
    if (flags != 0u) {
      rec[nrec * kThreads] = (uint16_t)(((uint32_t)g << 8) | flags);
      ++nrec;
      got += __popc(flags);
    }
  }
  return got;
}

// Rare: fewer than E+1 members in the query's row; scan the library, keeping the
// E+1 smallest (distance, index) keys.
template <int E>
__device__ __noinline__ void library_search(const float* sj, const int32_t* order,
                                            const uint32_t* bits, int words, int off, int tau, int W,
                                            int n_m, int m, float (&dd)[E + 1], int (&nb)[E + 1]) {
  float q[E];
#pragma unroll
  for (int e = 0; e < E; ++e) q[e] = sj[m + off - e * tau];
  float kd[E + 1];
  int kl[E + 1];
#pragma unroll
  for (int s2 = 0; s2 <= E; ++s2) {
    kd[s2] = INFINITY;
    kl[s2] = INT_MAX;
  }
  for (int w = 0; w < words; ++w) {
    for (uint32_t left = bits[w]; left != 0u; left &= left - 1u) {
      const int l = order[32 * w + __ffs(left) - 1];
      if (abs(l - m) <= W) continue;
      const float d = d2_point<E>(sj, off, tau, q, l);
      if (key_less(d, l, kd[E], kl[E])) {
        int s2 = E;
        while (s2 > 0 && key_less(d, l, kd[s2 - 1], kl[s2 - 1])) {
          kd[s2] = kd[s2 - 1];
          kl[s2] = kl[s2 - 1];
          --s2;
        }
        kd[s2] = d;
        kl[s2] = l;
      }
    }
  }
#pragma unroll
  for (int s2 = 0; s2 <= E; ++s2) {
    nb[s2] = min(max(kl[s2], 0), n_m - 1);  // in bounds however few points qualified
    dd[s2] = sqrt_hw(kd[s2]);
  }
}

template <int E, bool kLanes, bool kStats>
__device__ void process_table_item(const KnnParams& p, const UnitDesc& u, int tile0,
                                   unsigned char* smem, RingMeta* meta, int& ring_n) {
  constexpr int K = E + 1;
  const int tid = threadIdx.x;
  const int n_m = u.n_m, tau = u.tau, stride = u.table_R, W = u.theiler;
  const int off = (E - 1) * tau;
  const float* sj = p.series + u.series_off + (int64_t)u.j * u.n;
  const int32_t* order = p.order + u.order_off;
  float* s_ring = reinterpret_cast<float*>(smem);
  uint16_t* s_rec = reinterpret_cast<uint16_t*>(smem + kRingBytes);  // [K][kThreads]
  uint32_t* s_bits = reinterpret_cast<uint32_t*>(smem + kRingBytes + kRecBytes);
  u64* s_keep = reinterpret_cast<u64*>(smem + p.lane_scratch);
  const int words = (n_m + 31) >> 5;
  __syncthreads();  // the previous item's readers of the bits are done
  for (int w = tid; w < (n_m + 32) >> 5; w += kThreads)  // one beyond the last position at least
    s_bits[w] = w < words ? p.bits[u.bits_off + w] : 0u;
  __syncthreads();

  const int tile1 = min(u.n_tiles, tile0 + kTableChunk);
  for (int tile = tile0; tile < tile1; ++tile) {
    const int pos = tile * kQT + tid;
    const bool valid = pos < n_m;
    const int m = order[valid ? pos : n_m - 1];
    const int64_t row = u.table_off + (int64_t)(valid ? pos : 0) * stride;
    uint32_t st_entries = 0;
    uint16_t* rec = s_rec + tid;
    const int got =
        p.table_u16 ? table_walk<K, uint16_t, kStats>(static_cast<const uint16_t*>(p.table) + row,
                                                      order, stride >> 3, m, W, s_bits, rec, valid,
                                                      st_entries)
                    : table_walk<K, int32_t, kStats>(static_cast<const int32_t*>(p.table) + row,
                                                     order, stride >> 3, m, W, s_bits, rec, valid,
                                                     st_entries);
    const bool full = got >= K;
    if (kStats) {
      const uint32_t ent = __reduce_add_sync(kFull, st_entries);
      const unsigned vq = __popc(__ballot_sync(kFull, valid));
      const unsigned fb = __popc(__ballot_sync(kFull, valid && !full));
      if ((tid & 31) == 0) {
        atomicAdd(&p.stats[kStatTableEntries], (unsigned long long)ent);
        atomicAdd(&p.stats[kStatTableQueries], (unsigned long long)vq);
        if (fb) atomicAdd(&p.stats[kStatTableFallbacks], (unsigned long long)fb);
      }
    }
    int nb[E + 1];
    float dd[E + 1];
    if (full) {
      // the first E+1 flagged ranks; their points and distances are read from
      // the table (the stored distances are the bits the epilogue would
      // compute: the build used the same rounding sequence and square root)
      int ri = 0;
      uint32_t cur = rec[0];
#pragma unroll
      for (int s2 = 0; s2 <= E; ++s2) {
        if ((cur & 0xffu) == 0u) cur = rec[(++ri) * kThreads];
        const int c = __ffs(cur & 0xffu) - 1;
        cur &= ~(1u << c);
        const int64_t at = row + 8 * (int)(cur >> 8) + c;
        dd[s2] = p.table_pairs ? __ldg(reinterpret_cast<const float2*>(p.table_dist) + at).x
                               : __ldg(p.table_dist + at);
        nb[s2] = order[p.table_u16 ? (int)__ldg(static_cast<const uint16_t*>(p.table) + at)
                                   : __ldg(static_cast<const int32_t*>(p.table) + at)];
      }
    } else if (!valid) {
#pragma unroll
      for (int s2 = 0; s2 <= E; ++s2) {
        dd[s2] = 0.f;
        nb[s2] = 0;
      }
    } else {
      library_search<E>(sj, order, s_bits, words, off, tau, W, n_m, m, dd, nb);
    }
    finish_tile<E, kLanes, false, true>(p, u, tile, m, valid, dd, nb, s_ring, meta, ring_n, s_keep);
  }
}

// kMinCtas CTAs per SM: two (128 registers) with a lane per target, whose
// epilogue is the work; four (64 registers) else, where the walk waits on L2.
template <int E, bool kLanes, bool kStats, int kMinCtas>
__global__ void __launch_bounds__(kThreads, kMinCtas) knn_table_kernel(KnnParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  __shared__ RingMeta s_meta[kRing];
  int ring_n = 0;  // staged prediction vectors (the same in every thread)
  chain_begin();
  for (int64_t round = 0;; ++round) {
    if (p.persistent) {
      if (threadIdx.x == 0) s_item = (int)atomicAdd(p.item_counter, 1u);
      __syncthreads();
    }
    const int it = p.persistent ? s_item : (round == 0 ? (int)blockIdx.x : INT_MAX);
    __syncthreads();
    if ((int64_t)it >= p.n_items) break;
    const WorkItem w = p.items[it];
    const UnitDesc u = p.units[w.unit];
    if (u.E != E || lane_per_target(u) != kLanes) {
      if (threadIdx.x == 0) atomicOr(p.err, kErrBadUnit);
      continue;
    }
    process_table_item<E, kLanes, kStats>(p, u, w.tile, smem, s_meta, ring_n);
  }
  if (ring_n > 0) flush_ring(p, reinterpret_cast<const float*>(smem), s_meta, ring_n);
}

// kPrune false (E <= 2): for manifolds in time order, where no pair can be excluded.
template <int E, bool kLanes, bool kStats, bool kPrune = true>
__global__ void __launch_bounds__(kThreads, 3) knn_fused_kernel(KnnParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  __shared__ float2 s_qbox[kThreads / 32 * kBoxDims];
  __shared__ RingMeta s_meta[kRing];
  int ring_n = 0;  // staged prediction vectors (the same in every thread)
  chain_begin();
  for (int64_t round = 0;; ++round) {
    if (p.persistent) {
      if (threadIdx.x == 0) s_item = (int)atomicAdd(p.item_counter, 1u);
      __syncthreads();
    }
    const int it = p.persistent ? s_item : (round == 0 ? (int)blockIdx.x : INT_MAX);
    __syncthreads();
    if ((int64_t)it >= p.n_items) break;
    const WorkItem w = p.items[it];
    const UnitDesc u = p.units[w.unit];
    if (u.E != E || lane_per_target(u) != kLanes) {
      if (threadIdx.x == 0) atomicOr(p.err, kErrBadUnit);
      continue;
    }
    if (p.variant[E] == 1)
      process_item<E, 1, kLanes, kStats, kPrune>(p, u, w.tile, w.count, smem, s_meta, s_qbox, ring_n);
    else
      process_item<E, 0, kLanes, kStats, kPrune>(p, u, w.tile, w.count, smem, s_meta, s_qbox, ring_n);
  }
  if (ring_n > 0)
    flush_ring(p, reinterpret_cast<const float*>(smem + kCoordBytes + kBufBytes), s_meta, ring_n);
}

// Ring, records and bits: every manifold of the launch fits.
size_t table_base_smem(int max_nm) {
  const size_t bits = (size_t)((max_nm + 32) / 32) * 4;
  return ((size_t)kRingBytes + (size_t)kRecBytes + bits + 15) / 16 * 16;
}
size_t table_smem(int max_nm, bool lane_targets) {
  return table_base_smem(max_nm) +
         (lane_targets ? (size_t)(kMaxE + 1) * kThreads * 8 + kLaneScratch : 0);
}

}  // namespace

// The kernels of one E, in a translation unit of their own (CCM_E).
template <int E>
cudaError_t KnnKernels<E>::launch(const KnnParams& p, bool lanes, int grid, LaunchStream s) {
  if constexpr (E <= 2)
    if (!p.prune && !lanes && !p.stats)
      return launch_chained(knn_fused_kernel<E, false, false, false>, dim3((unsigned)grid), kThreads,
                            kSmemBytes, s, p);
  const auto fn = lanes ? (p.stats ? knn_fused_kernel<E, true, true> : knn_fused_kernel<E, true, false>)
                        : (p.stats ? knn_fused_kernel<E, false, true> : knn_fused_kernel<E, false, false>);
  return launch_chained(fn, dim3((unsigned)grid), kThreads, kSmemBytes, s, p);
}

template <int E>
cudaError_t KnnKernels<E>::prepare() {
  for (const auto fn : {knn_fused_kernel<E, false, false>, knn_fused_kernel<E, false, true>,
                        knn_fused_kernel<E, true, false>, knn_fused_kernel<E, true, true>}) {
    const cudaError_t e =
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
    if (e != cudaSuccess) return e;
  }
  if constexpr (E <= 2)
    return cudaFuncSetAttribute(knn_fused_kernel<E, false, false, false>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  return cudaSuccess;
}

template <int E>
cudaError_t KnnKernels<E>::occupancy(int* ctas) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, knn_fused_kernel<E, false, false>,
                                                       kThreads, kSmemBytes);
}

template <int E>
static auto table_kernel(bool lanes, bool stats) {
  if (lanes) return stats ? knn_table_kernel<E, true, true, 2> : knn_table_kernel<E, true, false, 2>;
  return stats ? knn_table_kernel<E, false, true, 4> : knn_table_kernel<E, false, false, 4>;
}

template <int E>
cudaError_t KnnKernels<E>::launch_table(const KnnParams& params, int max_nm, bool lanes, int grid,
                                        LaunchStream s) {
  KnnParams p = params;
  p.lane_scratch = (int32_t)table_base_smem(max_nm);
  return launch_chained(table_kernel<E>(lanes, p.stats != nullptr), dim3((unsigned)grid), kThreads,
                        table_smem(max_nm, lanes), s, p);
}

template <int E>
cudaError_t KnnKernels<E>::prepare_table() {
  // the largest bitmap any plan may need (manifolds up to kTableMaxNm points);
  // set once, so that plans of different sizes never lower it for each other
  for (const auto fn : {knn_table_kernel<E, false, false, 4>, knn_table_kernel<E, false, true, 4>,
                        knn_table_kernel<E, true, false, 2>, knn_table_kernel<E, true, true, 2>}) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)table_smem(kTableMaxNm, true));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int E>
cudaError_t KnnKernels<E>::occupancy_table(int max_nm, bool lanes, int* ctas) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, table_kernel<E>(lanes, false),
                                                       kThreads, table_smem(max_nm, lanes));
}

template struct KnnKernels<CCM_E>;

}  // namespace ccm
