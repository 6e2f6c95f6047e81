// Table scan of units with one target: up to 32 realizations of one (library
// variable, target, E, tau) are served by one walk of each query's row of the
// distance indexing table (table.cu; compiled once per E).
//
// A warp owns a query and a lane a realization.  The row holds the query's
// nearest manifold points, nearest first, as positions of the query order.  In
// a step the lanes read 32 consecutive ranks (one coalesced access), look up
// the membership word of each (bit r: realization r's library holds the point)
// and transpose the 32 x 32 bits across the warp, so that every lane holds the
// members of its own realization among the 32 ranks.  A lane that still lacks
// neighbours records the step's mask (at most E+1 records: each holds a
// member); the walk ends when every lane has E+1.  Then each lane reads off its
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
// Bound: issue (57 %) and the latency of the row and pair loads behind the
// shuffles (ncu, E = 10).  Sweep (N = 10^4, E = 1..10, L = 142..9000, r = 250):
// 65 ms a run; a thread per query and four realizations per walk 151 ms.  Two
// variables of N = 10^5 (E = 3..6, L = 5000..50000): 18 ms, before 109 ms.
#include <limits.h>
#include <math.h>

#include "bits.cuh"
#include "ccm_internal.h"
#include "launch.cuh"
#include "moments.cuh"

namespace ccm {
namespace {

using u64 = unsigned long long;

constexpr int kScanThreads = 512;
constexpr int kScanWarps = kScanThreads / 32;
constexpr int kQueriesPerWarp = kQT / kScanWarps;
// A realization's predictions of a tile (vec_slot order).  The odd stride
// spreads the 32 lanes' stores of one query over the banks.
constexpr int kScanVec = kQT + 9;

template <int E>
constexpr size_t scan_fixed_smem() {
  return 32 * kScanVec * 4 + (size_t)(E + 1) * kScanThreads * (4 + 2);
}

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

// Weights and prediction (paper Sect. 2.1) from the E+1 distances and target
// values, nearest first: the brute-force epilogue's operations in its order.
template <int E>
__device__ __forceinline__ float predict(const float (&d)[E + 1], const float (&v)[E + 1],
                                         float wfloor) {
  const float d1 = d[0];
  const float inv_d1 = (d1 > 0.f) ? rcp_hw(d1) : 0.f;
  float w[E + 1];
#pragma unroll
  for (int s = 0; s <= E; ++s) w[s] = simplex_exp(d[s], inv_d1);
  if (!(d1 > 0.f)) {  // rare: the nearest at distance 0
#pragma unroll
    for (int s = 0; s <= E; ++s) w[s] = simplex_limit(d[s]);
  }
  float usum = 0.f, acc = 0.f;
#pragma unroll
  for (int s = 0; s <= E; ++s) {
    w[s] = fmaxf(w[s], wfloor);
    usum = __fadd_rn(usum, w[s]);
    acc = __fmaf_rn(w[s], v[s], acc);
  }
  return __fmul_rn(acc, rcp_hw(usum));
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
      for (int i = tid; i < quads; i += kScanThreads) dst[i] = __ldg(src + i);
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
      const float scale = p.obs_stat[tg.obs_tile + tile].scale;
      const int nq = min(kQT, n_m - tile * kQT);
      for (int i = 0; i < kQueriesPerWarp; ++i) {
        const int q = warp * kQueriesPerWarp + i;
        if (q >= nq) break;
        const int pos = tile * kQT + q;
        const int64_t row = u.table_off + (int64_t)pos * stride;
        const int m = kGeneral ? order[pos] : 0;
        // the walk: lane l holds rank 31 - l of a step, so that the highest set
        // bit of a realization's mask is its nearest member
        const Index* ip = static_cast<const Index*>(p.table) + row + (31 - lane);
        const Index* const end = ip + stride;
        int got = 0, recs = 0, c = 0;
        auto lookup = [&](uint32_t x) {
          uint32_t word = kSmemWords ? s_words[x] : __ldg(words + x);
          if (kGeneral && W > 0 && word != 0u) {  // points inside the exclusion window
            const int l = order[x];
            if ((unsigned)l - (unsigned)m + (unsigned)W <= 2u * (unsigned)W) word = 0u;
          }
          return word;
        };
        auto record = [&](uint32_t members) {
          if (members != 0u && got < K) {
            mask[recs * kScanThreads] = members;
            step[recs * kScanThreads] = (uint16_t)c;
            ++recs;
            got += __popc(members);
          }
          ++c;
        };
        uint32_t xa = (uint32_t)__ldg(ip);
        if (dense) {  // 32 ranks a step: the first ones mostly suffice
          for (;;) {
            const uint32_t wa = lookup(xa);
            ip += 32;
            const bool more = ip < end;
            if (more) xa = (uint32_t)__ldg(ip);
            record(tr(wa));
            if (!more || !__any_sync(kAllLanes, mine && got < K)) break;
          }
        } else {  // 64 ranks a step, the next step's loads in flight
          uint32_t xb = (uint32_t)__ldg(ip + 32);
          for (;;) {
            const uint32_t wa = lookup(xa), wb = lookup(xb);
            ip += 64;
            const bool more = ip < end;
            if (more) {
              xa = (uint32_t)__ldg(ip);
              xb = (uint32_t)__ldg(ip + 32);
            }
            const uint32_t ma = tr(wa), mb = tr(wb);
            record(ma);
            record(mb);
            if (!more || !__any_sync(kAllLanes, mine && got < K)) break;
          }
        }
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
          uint32_t cur = mask[0];
          int base = step[0] * 32, rec = 0;
#pragma unroll
          for (int s = 0; s < K; ++s) {
            if (cur == 0u) {
              ++rec;
              cur = mask[rec * kScanThreads];
              base = step[rec * kScanThreads] * 32;
            }
            const int b = __clz(cur);
            cur ^= 0x80000000u >> b;
            rank[s] = base + b;
          }
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
        s_vec[lane * kScanVec + vec_slot(q)] = __fmul_rn(y, scale);
      }
      __syncthreads();
      // two vectors a warp: half a warp's lane g sums the tile's queries 16g ..
      // 16g+15 as two groups, then the tree (the order of tile_sums_warp)
      const int vec = warp * 2 + (lane >> 4), g = lane & 15;
      if (warp * 2 < count) {
        const int64_t rec = tg.obs_tile + tile;
        const float* ys = s_vec + vec * kScanVec;
        const float2* a = p.obs + rec * kQT;
        const float c0 = ys[0];
        const packed cc = pack2(c0, c0);
        TileSums2 both = zero_sums2();
#pragma unroll 4
        for (int i = 0; i < kMomentGroup; ++i) {
          const int qa = 16 * g + i, qb = qa + kMomentGroup;
          const float ya = ys[vec_slot(qa)], yb = ys[vec_slot(qb)];
          add_query2(both, pack2(qa < nq ? ya : c0, qb < nq ? yb : c0), __ldg(a + obs_slot(qa)),
                     __ldg(a + obs_slot(qb)), cc);
        }
        TileSums half[2];
        unpack_sums(both, half[0], half[1]);
        TileSums m = merge_sums(half[0], half[1]);
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) m = merge_across(m, o);
        if (g == 0 && vec < count)
          store_sums(p.partials + 2 * (p.units[w.unit + vec].part_off + tile), c0, m);
      }
      __syncthreads();
    }
  }
}

template <int E>
size_t scan_smem(int max_nm, bool smem_words) {
  return scan_fixed_smem<E>() + (smem_words ? (size_t)member_words(max_nm) * 4 : 0);
}

// The membership words go to shared memory while two CTAs still fit an SM;
// beyond that the words' spatial coherence in L1 serves better than half the
// warps.
template <int E>
bool words_in_smem(int max_nm) {
  return scan_smem<E>(max_nm, true) <= kScanSmemMax;
}

template <int E>
auto scan_variant(int max_nm, bool u16, bool general) {
  const bool sm = words_in_smem<E>(max_nm);
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
  const bool sm = p.table_u16 && words_in_smem<E>(max_nm);
  return launch_chained(scan_variant<E>(max_nm, p.table_u16 != 0, general), dim3((unsigned)grid),
                        kScanThreads, scan_smem<E>(max_nm, sm), s, p);
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

template struct KnnKernels<CCM_E>;

}  // namespace ccm
