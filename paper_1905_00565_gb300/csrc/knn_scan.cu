// Table scan in groups of realizations: up to 32 realizations of one (library
// variable, E, tau) are served by one walk of each query's row of the distance
// indexing table (table.cu; compiled once per E).  scan_kernel: units with one
// target; group_kernel: units with many.
//
// A warp owns a query and a lane a realization (the walk: row_walk.cuh).  When
// every lane has met E+1 members of its library, each reads off its
// first E+1 ranks, loads their (distance, target value) pairs from the same
// row, and forms the weights and the prediction, in the order and with the
// operations of the brute-force epilogue: every bit of rho is the same.
//
// Predictions go to a shared-memory vector per realization; after a tile of
// 256 queries the warps reduce the vectors' moments (moments.cuh).
//
// Why this mapping: a row is read once for 32 realizations, sequentially, and
// the lanes' pair loads fall into the same few kilobytes.  With a thread per
// query and four realizations per walk every load of a warp touched 32 rows,
// the walk waited on L2 (6 stalls per issue), and it ran until the slowest of
// 128 (query, realization) was done.
//
// Bound: issue (64 %) and the latency of the row and pair loads behind the
// shuffles (ncu, E = 10).  Sweep (N = 10^4, E = 1..10, r = 250), libraries from
// 142 points on: 151 ms with a thread per query and four realizations a walk,
// 65 with this mapping; now that libraries from 100 points on read tables 97.
// Two variables of N = 10^5 (E = 3..6, L = 1000..50000; before from L = 5000 on):
// 109 -> 31 ms.
#include <limits.h>
#include <math.h>

#include <type_traits>

#include "ccm_internal.h"
#include "launch.cuh"
#include "moments.cuh"
#include "row_walk.cuh"

namespace ccm {
namespace {

using u64 = unsigned long long;

constexpr int kScanWarps = kScanThreads / 32;
constexpr int kQueriesPerWarp = kQT / kScanWarps;

// A realization with fewer than E+1 members in the row (rare): the warp scans
// its whole library, every lane keeping the E+1 smallest keys of its words'
// members, four members' loads in flight (the loads' latency is the cost: the
// other warps of the tile wait).  keys[s] = (bits of the squared distance,
// manifold index), for every lane.
template <int E>
__device__ __noinline__ void search_library(const KnnParams& p, const UnitDesc& u, int r, int m,
                                            u64 (&keys)[E + 1]) {
  const int lane = threadIdx.x & 31;
  const int n_m = u.n_m, tau = u.tau, off = (E - 1) * tau, W = u.theiler;
  const int words = (n_m + 31) >> 5;
  const uint32_t* bits = p.bits + u.bits_off + (int64_t)r * words;
  const int32_t* order = p.order + u.order_off;
  const float* s = p.series + u.series_off + (int64_t)u.j * u.n + off;
  float q[E];
#pragma unroll
  for (int e = 0; e < E; ++e) q[e] = s[m - e * tau];
  u64 mine[E + 1];  // ascending
#pragma unroll
  for (int k = 0; k <= E; ++k) mine[k] = ~0ull;
  int w = lane;
  uint32_t left = w < words ? bits[w] : 0u;
  for (;;) {
    int x[4], got = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      while (left == 0u && w < words) {
        w += 32;
        left = w < words ? bits[w] : 0u;
      }
      x[c] = m;
      if (left != 0u) {
        x[c] = order[w * 32 + __ffs(left) - 1];
        left &= left - 1u;
        ++got;
      }
    }
    if (got == 0) break;
    float acc[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float diff = __fsub_rn(q[0], s[x[c]]);
      acc[c] = __fmul_rn(diff, diff);
#pragma unroll
      for (int e = 1; e < E; ++e) {
        diff = __fsub_rn(q[e], s[x[c] - e * tau]);
        acc[c] = __fmaf_rn(diff, diff, acc[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const u64 key = ((u64)__float_as_uint(acc[c]) << 32) | (uint32_t)x[c];
      if (c < got && abs(x[c] - m) > W && key < mine[E]) {
#pragma unroll
        for (int k = E; k > 0; --k)
          mine[k] = key < mine[k - 1] ? mine[k - 1] : (key < mine[k] ? key : mine[k]);
        mine[0] = key < mine[0] ? key : mine[0];
      }
    }
  }
  __syncwarp();
#pragma unroll
  for (int k = 0; k <= E; ++k) {
    u64 best = mine[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const u64 y = __shfl_xor_sync(kAllLanes, best, o);
      best = y < best ? y : best;
    }
    keys[k] = best;
    if (mine[0] == best) {
#pragma unroll
      for (int i = 0; i < E; ++i) mine[i] = mine[i + 1];
      mine[E] = ~0ull;
    }
  }
}

// Simplex weights (paper Sect. 2.1) of the E+1 distances, nearest first, and
// their sum: the brute-force epilogue's operations in its order.
template <int E>
__device__ __forceinline__ float simplex_weights(const float (&d)[E + 1], float wfloor,
                                                 float (&w)[E + 1]) {
  const float d1 = d[0];
  const float inv_d1 = (d1 > 0.f) ? rcp_hw(d1) : 0.f;
#pragma unroll
  for (int s = 0; s <= E; ++s) w[s] = simplex_exp(d[s], inv_d1);
  if (!(d1 > 0.f)) {  // rare: the nearest at distance 0
#pragma unroll
    for (int s = 0; s <= E; ++s) w[s] = simplex_limit(d[s]);
  }
  float usum = 0.f;
#pragma unroll
  for (int s = 0; s <= E; ++s) {
    w[s] = fmaxf(w[s], wfloor);
    usum = __fadd_rn(usum, w[s]);
  }
  return usum;
}

template <int E>
__device__ __forceinline__ float predict(const float (&d)[E + 1], const float (&v)[E + 1],
                                         float wfloor) {
  float w[E + 1];
  const float usum = simplex_weights<E>(d, wfloor, w);
  float acc = 0.f;
#pragma unroll
  for (int s = 0; s <= E; ++s) acc = __fmaf_rn(w[s], v[s], acc);
  return __fmul_rn(acc, rcp_hw(usum));
}

__device__ __noinline__ void exact_vector(const TileTarget t, const float* ys, float4* part) {
  exact_sums_warp(t, ys, part);
}

// kSmemWords: the item's membership words lie in shared memory (else they are
// read from global memory, spatially coherent in query order and so mostly
// from L1).  kGeneral: with an exclusion window, search counters, or neighbour
// lists and predictions returned.
template <int E, typename Index, bool kSmemWords, bool kGeneral>
__global__ void __launch_bounds__(kScanThreads, 2) scan_kernel(KnnParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  constexpr int K = E + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* s_vec = reinterpret_cast<float*>(smem);                             // [32][kScanVec]
  uint32_t* s_mask = reinterpret_cast<uint32_t*>(s_vec + 32 * kScanVec);     // [K][kScanThreads]
  uint16_t* s_step = reinterpret_cast<uint16_t*>(s_mask + K * kScanThreads); // [K][kScanThreads]
  uint32_t* s_words = reinterpret_cast<uint32_t*>(s_step + K * kScanThreads);
  const BitTranspose tr(lane);
  chain_begin();
  for (int round = 0;; ++round) {
    if (p.persistent && tid == 0) s_item = (int)atomicAdd(p.item_counter, 1u);
    __syncthreads();
    const int it = p.persistent ? s_item : (round == 0 ? (int)blockIdx.x : INT_MAX);
    if ((int64_t)it >= p.n_items) break;
    const WorkItem w = p.items[it];
    const UnitDesc& u = p.units[w.unit];  // the realizations' common description
    const int count = w.count & 0xff, tile0 = w.tile, n_m = u.n_m, stride = u.table_R;
    const int tile1 = min(u.n_tiles, tile0 + (w.count >> 8));
    const int W = u.theiler;
    if (u.E != E || u.n_targets != 1 || count < 1 || count > 32) {
      if (tid == 0) atomicOr(p.err, kErrBadUnit);
      __syncthreads();
      continue;
    }
    const uint32_t* words = p.words + u.words_off;
    if (kSmemWords) {
      const int quads = member_words(n_m) >> 2;
      const uint4* src = reinterpret_cast<const uint4*>(words);
      uint4* dst = reinterpret_cast<uint4*>(s_words);
      for (int i = tid; i < quads; i += kScanThreads) dst[i] = src[i];
    }
    __syncthreads();
    const int32_t* order = p.order + u.order_off;
    const TargetDesc& tg = p.targets[u.tgt_off];
    const bool mine = lane < count;
    // expected ranks walked, with the spread of the slowest of 32 realizations
    const bool dense = 2 * K * (int64_t)n_m <= 32 * (int64_t)u.L;
    uint32_t* mask = s_mask + tid;
    uint16_t* step = s_step + tid;
    for (int tile = tile0; tile < tile1; ++tile) {
      const SeriesScale sc = p.obs_stat[tg.obs_tile + tile].series;
      const int nq = min(kQT, n_m - tile * kQT);
      for (int i = 0; i < kQueriesPerWarp; ++i) {
        const int q = warp * kQueriesPerWarp + i;
        if (q >= nq) break;
        const int pos = tile * kQT + q;
        const int64_t row = u.table_off + (int64_t)pos * stride;
        const int m = kGeneral ? order[pos] : 0;
        int c;
        const int got = group_walk<K, kScanThreads, Index, kGeneral>(
            static_cast<const Index*>(p.table) + row, stride, dense, mine, kSmemWords ? s_words : words,
            order, m, W, tr, mask, step, c);
        const bool full = mine && got >= K;
        if (kGeneral && p.stats) {
          const unsigned shorts = __popc(__ballot_sync(kAllLanes, mine && !full));
          if (lane == 0) {
            atomicAdd(&p.stats[kStatTableQueries], (unsigned long long)count);
            atomicAdd(&p.stats[kStatTableEntries], 32ull * c);
            if (shorts) atomicAdd(&p.stats[kStatTableFallbacks], (unsigned long long)shorts);
          }
        }
        float y = 0.f;
        if (full) {
          int rank[K];
          first_ranks<K, kScanThreads>(mask, step, rank);
          const float2* dv = reinterpret_cast<const float2*>(p.table_dist) + row;
          float d[K], v[K];
#pragma unroll
          for (int s = 0; s < K; ++s) {
            const float2 f = __ldg(dv + rank[s]);
            d[s] = f.x;
            v[s] = f.y;
          }
          y = predict<E>(d, v, u.wfloor);
          if (kGeneral && p.dbg_nbr) {
            int32_t* out = p.dbg_nbr + p.targets[u.tgt_off + lane].nbr_off + (int64_t)m * K;
#pragma unroll
            for (int s = 0; s < K; ++s)
              out[s] = order[static_cast<const Index*>(p.table)[row + rank[s]]];
          }
        }
        for (unsigned left = __ballot_sync(kAllLanes, mine && !full); left; left &= left - 1u) {
          const int r = __ffs(left) - 1;
          const int qm = order[pos];
          u64 keys[K];
          search_library<E>(p, u, r, qm, keys);
          const float* si = p.series + u.series_off + (int64_t)tg.i * u.n + (E - 1) * u.tau;
          float d[K], v[K];
          int nb[K];
#pragma unroll
          for (int s = 0; s < K; ++s) {
            // in bounds however few points qualified
            nb[s] = min(max((int)(uint32_t)keys[s], 0), n_m - 1);
            d[s] = sqrt_hw(__uint_as_float((uint32_t)(keys[s] >> 32)));
            v[s] = si[nb[s]];
          }
          const float yr = predict<E>(d, v, u.wfloor);
          if (lane == r) {
            y = yr;
            if (kGeneral && p.dbg_nbr) {
              int32_t* out = p.dbg_nbr + p.targets[u.tgt_off + r].nbr_off + (int64_t)m * K;
#pragma unroll
              for (int s = 0; s < K; ++s) out[s] = nb[s];
            }
          }
        }
        if (kGeneral && p.dbg_xhat && mine) p.dbg_xhat[p.targets[u.tgt_off + lane].q_off + m] = y;
        s_vec[lane * kScanVec + vec_slot(q)] = y;
      }
      __syncthreads();
      // two vectors a warp: half a warp's lane g sums the tile's queries 16g ..
      // 16g+15 as two groups, then the tree (the order of tile_sums_warp)
      const int vec = warp * 2 + (lane >> 4), g = lane & 15;
      if (warp * 2 < count) {
        const int64_t rec = tg.obs_tile + tile;
        const float* ys = s_vec + vec * kScanVec;
        const float2* a = p.obs + rec * kQT;
        const ObsStat* stat = p.obs_stat + rec;
        const float scale = sc.scale, c0 = __fmul_rn(ys[0], scale);
        const packed cc = pack2(c0, c0), ss = pack2(scale, scale);
        TileSums2 both = zero_sums2();
#pragma unroll 4
        for (int i = 0; i < kMomentGroup; ++i) {
          const int qa = 16 * g + i, qb = qa + kMomentGroup;
          const float ya = ys[vec_slot(qa)], yb = ys[vec_slot(qb)];
          add_query2(both, mul2(pack2(qa < nq ? ya : ys[0], qb < nq ? yb : ys[0]), ss),
                     __ldg(a + obs_slot(qa)), __ldg(a + obs_slot(qb)), cc);
        }
        TileSums half[2];
        unpack_sums(both, half[0], half[1]);
        TileSums m = merge_sums(half[0], half[1]);
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) m = merge_across(m, o);
        const bool writes = g == 0 && vec < count, redo_mine = writes && too_small(m.b2.h, sc);
        if (writes && !redo_mine)
          store_sums(p.partials + 2 * (p.units[w.unit + vec].part_off + tile), c0, m);
        for (unsigned redo = __ballot_sync(kAllLanes, redo_mine); redo; redo &= redo - 1u) {
          const int v = warp * 2 + (__ffs(redo) > 16 ? 1 : 0);
          exact_vector(TileTarget{p.series + u.series_off + (int64_t)tg.i * u.n + (E - 1) * u.tau,
                                  order + tile * kQT, stat, nq},
                       s_vec + v * kScanVec,
                       p.partials + 2 * (p.units[w.unit + v].part_off + tile));
        }
      }
      __syncthreads();
    }
  }
}

// Units with many targets, up to lane_group(E) realizations of one (library
// variable, E, tau) and one query tile an item.  Phase 1: a warp walks a query's
// row for all of them at once, a lane a realization, and leaves each one's
// weights and neighbours (byte offsets into the time-major series) in shared
// memory.  Phase 2: a team of four warps takes a realization and 32 targets, a
// lane a target and a quarter of the tile's queries a warp: a neighbour's values
// of 32 targets are one coalesced read, the moments stay in the lane's registers
// and meet once per task.
//
// Bound: issue (50 %) and the latency of the series reads (half an SM's warps
// at 80 registers; 64 and 128 registers are slower).  A realization at a time
// per CTA, every thread walking its own row, left 32 lines per load of a row's
// entries and two block barriers per 32 targets: 64 variables, N = 5000, E =
// 2..4, r = 25, L = 296 .. 4500, all pairs 42.5 ms, now 34.3.  Teams rather than
// a warp a task: 16 to 40 tasks do not divide among 24 warps (24 variables 0.82
// -> 0.76 ms).  160 KB for the realizations rather than 128: 35.0 -> 34.3.
constexpr int kGroupThreads = 768;
constexpr int kTeam = 4;  // warps a (realization, 32 targets): a quarter of the tile each
constexpr int kTeamQueries = kQT / kTeam;
static_assert(kGroupThreads % (32 * kTeam) == 0 && kTeamQueries % (2 * kMomentGroup) == 0, "teams");
static_assert(4 * kGroupThreads * 6 >= kGroupThreads / 32 * 6 * 32 * 4, "the teams' sums fit the records");
// A barrier of one team's warps (barrier 0 is the block's).
__device__ __forceinline__ void team_barrier(int team) {
  asm volatile("bar.sync %0, %1;" ::"r"(team + 1), "n"(32 * kTeam) : "memory");
}
template <int E>
constexpr int kKeepStride = (E + 1) * kQT + 1;  // entries a realization; odd: 32 lanes, 32 banks
template <int E>
__host__ __device__ constexpr size_t group_fixed_smem() {
  return (size_t)(lane_group(E) * kKeepStride<E> + 1) / 2 * 2 * 8 +
         (size_t)(lane_group(E) * (kQT + 1) + 3) / 4 * 16 +
         (size_t)(E + 1 < 4 ? 4 : E + 1) * kGroupThreads * (4 + 2);
}

// The prediction of query q from a realization's weights and neighbours.
template <int E>
__device__ __forceinline__ float group_prediction(const float2* keep, const float* rus,
                                                  const char* col, int q) {
  float acc = 0.f;
#pragma unroll
  for (int s = 0; s <= E; ++s) {
    const float2 k = keep[s * kQT + q];
    acc = __fmaf_rn(k.x, __ldg(reinterpret_cast<const float*>(col + __float_as_uint(k.y))), acc);
  }
  return __fmul_rn(acc, rus[q]);
}

// Whether this warp is the one of the task's team that stores its sums.
__device__ __forceinline__ bool stores_task(int task, int warp) {
  constexpr int kTeams = kGroupThreads / 32 / kTeam;
  return task % kTeams == warp / kTeam && task / kTeams % kTeam == warp % kTeam;
}

// Of the sums this lane stored, those whose predictions spread too little for them:
// again in FP64.
template <int E>
__device__ __noinline__ void exact_tasks(const float2* s_keep, const float* s_rus, const float* st,
                                         const TargetDesc* tgs, int T, int n_tiles, int nq, int count,
                                         const UnitDesc* units, float4* part, const float* x,
                                         int64_t n, const int32_t* order, const ObsStat* stat) {
  const int lane = threadIdx.x & 31;
  for (int task = 0; task < count * ((T + 31) / 32); ++task) {
    const int r = task % count, t = task / count * 32 + lane;
    if (!stores_task(task, threadIdx.x >> 5) || t >= T) continue;
    const TargetDesc& tg = tgs[t];
    float4* to = part + 2 * (units[r].part_off + (int64_t)t * n_tiles);
    if (!too_small(to->w, stat[tg.obs_tile].series)) continue;
    const float2* keep = s_keep + r * kKeepStride<E>;
    const float* rus = s_rus + r * (kQT + 1);
    const char* col = reinterpret_cast<const char*>(st + tg.i);
    exact_sums_lane(TileTarget{x + (int64_t)tg.i * n, order, stat + tg.obs_tile, nq},
                    [=](int q) { return group_prediction<E>(keep, rus, col, q); }, to);
  }
}

template <int E, bool kGeneral>
__global__ void __launch_bounds__(kGroupThreads, 1) group_kernel(KnnParams p) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_item;
  constexpr int K = E + 1, kWarps = kGroupThreads / 32, KS = kKeepStride<E>, G = lane_group(E);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float2* s_keep = reinterpret_cast<float2*>(smem);  // [realization][K][query]: weight, neighbour
  float* s_rus = reinterpret_cast<float*>(s_keep + (G * KS + 1) / 2 * 2);  // [realization][query]
  uint32_t* mask = reinterpret_cast<uint32_t*>(s_rus + (G * (kQT + 1) + 3) / 4 * 4) + tid;
  uint16_t* step = reinterpret_cast<uint16_t*>(mask - tid + K * kGroupThreads) + tid;
  uint32_t* s_words = reinterpret_cast<uint32_t*>(smem + group_fixed_smem<E>());
  const BitTranspose tr(lane);
  chain_begin();
  for (int round = 0;; ++round) {
    if (p.persistent && tid == 0) s_item = (int)atomicAdd(p.item_counter, 1u);
    __syncthreads();
    const int it = p.persistent ? s_item : (round == 0 ? (int)blockIdx.x : INT_MAX);
    if ((int64_t)it >= p.n_items) break;
    const WorkItem w = p.items[it];
    const int count = w.count, tile = w.tile;
    const UnitDesc& u = p.units[w.unit];  // the realizations' common description
    const int n_m = u.n_m, stride = u.table_R, W = u.theiler, T = u.n_targets;
    if (u.E != E || !lane_per_target(u) || count < 1 || count > G) {
      if (tid == 0) atomicOr(p.err, kErrBadUnit);
      __syncthreads();
      continue;
    }
    const uint32_t* words = p.words + u.words_off;
    if (p.group_words) {
      const uint4* src = reinterpret_cast<const uint4*>(words);
      uint4* dst = reinterpret_cast<uint4*>(s_words);
      for (int i = tid; i < member_words(n_m) >> 2; i += kGroupThreads) dst[i] = src[i];
    }
    __syncthreads();
    const int32_t* order = p.order + u.order_off;
    const int nq = min(kQT, n_m - tile * kQT);
    const bool mine = lane < count;
    const bool dense = 2 * K * (int64_t)n_m <= 32 * (int64_t)u.L;
    for (int q = warp; q < nq; q += kWarps) {
      const int pos = tile * kQT + q;
      const int64_t row = u.table_off + (int64_t)pos * stride;
      const int m = kGeneral ? order[pos] : 0;
      int c, got;
      auto walk = [&](auto* table, const uint32_t* from) {
        return group_walk<K, kGroupThreads, std::remove_const_t<std::remove_pointer_t<decltype(table)>>,
                          kGeneral>(table + row, stride, dense, mine, from, order, m, W, tr, mask,
                                    step, c);
      };
      if (!p.table_u16) got = walk(static_cast<const int32_t*>(p.table), words);
      else if (p.group_words) got = walk(static_cast<const uint16_t*>(p.table), s_words);
      else got = walk(static_cast<const uint16_t*>(p.table), words);
      const bool full = mine && got >= K;
      if (kGeneral && p.stats) {
        const unsigned shorts = __popc(__ballot_sync(kAllLanes, mine && !full));
        if (lane == 0) {
          atomicAdd(&p.stats[kStatTableQueries], (unsigned long long)count);
          atomicAdd(&p.stats[kStatTableEntries], 32ull * c);
          if (shorts) atomicAdd(&p.stats[kStatTableFallbacks], (unsigned long long)shorts);
        }
      }
      auto keep = [&](const float (&d)[K], const int (&nb)[K]) {
        float wt[K];
        const float usum = simplex_weights<E>(d, u.wfloor, wt);
#pragma unroll
        for (int s = 0; s < K; ++s)
          s_keep[lane * KS + s * kQT + q] = make_float2(wt[s], __uint_as_float((uint32_t)(nb[s] * u.st_stride) * 4u));
        s_rus[lane * (kQT + 1) + q] = rcp_hw(usum);
        if (kGeneral && p.dbg_nbr) {
          const int mq = order[pos];
          for (int t = 0; t < T; ++t)
            for (int s = 0; s < K; ++s)
              p.dbg_nbr[p.targets[p.units[w.unit + lane].tgt_off + t].nbr_off + (int64_t)mq * K + s] =
                  nb[s];
        }
      };
      if (full) {
        int rank[K], nb[K];
        float d[K];
        first_ranks<K, kGroupThreads>(mask, step, rank);
#pragma unroll
        for (int s = 0; s < K; ++s) {
          const int64_t at = row + rank[s];
          d[s] = p.table_pairs ? __ldg(reinterpret_cast<const float2*>(p.table_dist) + at).x
                               : __ldg(p.table_dist + at);
          nb[s] = order[p.table_u16 ? (int)__ldg(static_cast<const uint16_t*>(p.table) + at)
                                    : __ldg(static_cast<const int32_t*>(p.table) + at)];
        }
        keep(d, nb);
      }
      for (unsigned left = __ballot_sync(kAllLanes, mine && !full); left; left &= left - 1u) {
        const int r = __ffs(left) - 1;
        u64 keys[K];
        search_library<E>(p, u, r, order[pos], keys);
        float d[K];
        int nb[K];
#pragma unroll
        for (int s = 0; s < K; ++s) {
          // in bounds however few points qualified
          nb[s] = min(max((int)(uint32_t)keys[s], 0), n_m - 1);
          d[s] = sqrt_hw(__uint_as_float((uint32_t)(keys[s] >> 32)));
        }
        if (lane == r) keep(d, nb);
      }
    }
    __syncthreads();
    const float* st = p.st + u.st_off + (int64_t)(E - 1) * u.tau * u.st_stride;
    const TargetDesc* tgs = p.targets + u.tgt_off;
    const float2* obs = p.obs + tgs[0].obs_tile * kQT + (int64_t)tile * kQT * T;
    const int chunks = (T + 31) / 32;
    // [warp][value][lane], where the walks' records were
    float* sums = reinterpret_cast<float*>(mask - tid) + warp * 6 * 32 + lane;
    const int part = warp % kTeam, q0 = part * kTeamQueries;
    bool redo = false;
    for (int task = warp / kTeam; task < count * chunks; task += kWarps / kTeam) {
      const int chunk = task / count, r = task - chunk * count;
      const int t = min(chunk * 32 + lane, T - 1);  // lanes past the last target repeat it
      const TargetDesc& tg = tgs[t];
      const char* col = reinterpret_cast<const char*>(st + tg.i);
      const SeriesScale sc = p.obs_stat[tg.obs_tile + tile].series;
      const float scale = sc.scale;
      const float2* keep = s_keep + r * KS;
      const float* rus = s_rus + r * (kQT + 1);
      auto value = [&](int q) { return group_prediction<E>(keep, rus, col, q); };
      const float c = __fmul_rn(value(0), scale);
      const packed cc = pack2(c, c), ss = pack2(scale, scale);
      const float2* a = obs + t;
      // the tree's pending subtrees, indexed at run time: in local memory, not in the
      // loop's registers
      TileSums lv[3], sum;
      for (int n = 0; n < kTeamQueries / (2 * kMomentGroup); ++n) {  // 16 queries a turn
        const int qa = q0 + 2 * kMomentGroup * n, qb = qa + kMomentGroup;
        TileSums lo = zero_sums(), hi = zero_sums();
        if (qb + kMomentGroup <= nq && !(kGeneral && p.dbg_xhat)) {
          TileSums2 both = zero_sums2();
#pragma unroll 2
          for (int i = 0; i < kMomentGroup; ++i)
            add_query2(both, mul2(pack2(value(qa + i), value(qb + i)), ss),
                       __ldg(a + (int64_t)(qa + i) * T), __ldg(a + (int64_t)(qb + i) * T), cc);
          unpack_sums(both, lo, hi);
        } else {
          for (int q = qa; q < min(qb + kMomentGroup, nq); ++q) {
            const float y = value(q);
            if (kGeneral && p.dbg_xhat && chunk * 32 + lane < T)
              p.dbg_xhat[p.targets[p.units[w.unit + r].tgt_off + t].q_off + order[tile * kQT + q]] = y;
            add_query(q < qb ? lo : hi, __fmul_rn(y, scale), __ldg(a + (int64_t)q * T), c);
          }
        }
        sum = merge_sums(lo, hi);  // and up the tree of the tile's groups
        int l = 0;
        for (int up = n; up & 1; up >>= 1, ++l) sum = merge_sums(lv[l], sum);
        lv[l] = sum;
      }
      const float mine6[6] = {sum.b1.h, sum.b1.l, sum.b2.h, sum.b2.l, sum.ab.h, sum.ab.l};
#pragma unroll
      for (int x = 0; x < 6; ++x) sums[x * 32] = mine6[x];
      team_barrier(warp / kTeam);
      if (stores_task(task, warp) && chunk * 32 + lane < T) {
        auto load = [&](int i) {
          const float* f = sums + (i - part) * 6 * 32;
          TileSums m;
          m.b1 = Pair32{f[0], f[32]};
          m.b2 = Pair32{f[2 * 32], f[3 * 32]};
          m.ab = Pair32{f[4 * 32], f[5 * 32]};
          return m;
        };
        const TileSums m = merge_sums(merge_sums(load(0), load(1)), merge_sums(load(2), load(3)));
        store_sums(p.partials + 2 * (p.units[w.unit + r].part_off + (int64_t)t * u.n_tiles + tile), c, m);
        redo |= too_small(m.b2.h, sc);
      }
      team_barrier(warp / kTeam);
    }
    if (__builtin_expect(redo, 0))  // rare
      exact_tasks<E>(s_keep, s_rus, st, tgs, T, u.n_tiles, nq, count, p.units + w.unit,
                     p.partials + 2 * tile, p.series + u.series_off + (E - 1) * u.tau, u.n,
                     order + tile * kQT, p.obs_stat + tile);
    __syncthreads();
  }
}

// The membership words go to shared memory while two CTAs still fit an SM;
// beyond that the words' spatial coherence in L1 serves better than half the
// warps.
template <int E>
auto scan_variant(int max_nm, bool u16, bool general) {
  const bool sm = scan_words_in_smem(E, max_nm);
  if (u16) {
    if (general) return sm ? scan_kernel<E, uint16_t, true, true> : scan_kernel<E, uint16_t, false, true>;
    return sm ? scan_kernel<E, uint16_t, true, false> : scan_kernel<E, uint16_t, false, false>;
  }
  return general ? scan_kernel<E, int32_t, false, true> : scan_kernel<E, int32_t, false, false>;
}

}  // namespace

template <int E>
cudaError_t KnnKernels<E>::launch_scan(const KnnParams& p, int max_nm, int grid, LaunchStream s) {
  const bool general = p.window || p.stats || p.dbg_nbr || p.dbg_xhat;
  const size_t smem =
      scan_fixed_smem(E) +
      (p.table_u16 && scan_words_in_smem(E, max_nm) ? (size_t)member_words(max_nm) * 4 : 0);
  return launch_chained(scan_variant<E>(max_nm, p.table_u16 != 0, general), dim3((unsigned)grid),
                        kScanThreads, smem, s, p);
}

template <int E>
cudaError_t KnnKernels<E>::prepare_scan() {
  for (const auto fn : {scan_kernel<E, uint16_t, true, true>, scan_kernel<E, uint16_t, false, true>,
                        scan_kernel<E, uint16_t, true, false>, scan_kernel<E, uint16_t, false, false>,
                        scan_kernel<E, int32_t, false, true>, scan_kernel<E, int32_t, false, false>}) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kScanSmemMax);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int E>
cudaError_t KnnKernels<E>::launch_group(const KnnParams& params, int max_nm, int grid,
                                        LaunchStream s) {
  static_assert(group_fixed_smem<E>() <= kGroupSmemMax, "one CTA per SM");
  KnnParams p = params;
  const size_t with = group_fixed_smem<E>() + (size_t)member_words(max_nm) * 4;
  p.group_words = p.table_u16 && with <= kGroupSmemMax ? 1 : 0;
  const bool general = p.window || p.stats || p.dbg_nbr || p.dbg_xhat;
  return launch_chained(general ? group_kernel<E, true> : group_kernel<E, false>,
                        dim3((unsigned)grid), kGroupThreads,
                        p.group_words ? with : group_fixed_smem<E>(), s, p);
}

template <int E>
cudaError_t KnnKernels<E>::prepare_group() {
  for (const auto fn : {group_kernel<E, false>, group_kernel<E, true>}) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kGroupSmemMax);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template struct KnnKernels<CCM_E>;

}  // namespace ccm
