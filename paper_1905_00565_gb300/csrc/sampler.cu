// Library sampler: r random libraries of L manifold points, drawn without
// replacement (paper Sect. 1: r random subsamples of size L; Sect. 3.1: the
// pipeline input is a set of subsamples per (tau, E, L)).
//
// Random-key selection: manifold point m of unit (j, E, tau, L, k) gets the
// 64-bit key (v << 32) | m, where v is 32-bit half number m mod 8 of the
// Philox4x64-10 block at counter (floor(m/8), k, L, (j<<16)|(E<<8)|tau) under
// key (seed, 0), the halves numbered hi(w0), lo(w0), hi(w1), ..., lo(w3): one
// block gives the keys of eight consecutive points.  The library is the L
// points with the smallest keys, written in ascending m.  Keys are distinct,
// so the selection is a pure function of the counter.
//
// One CTA per unit.  The L-th smallest of N_m uniform keys lies within a few
// standard deviations of L/N_m, so one pass over the keys decides almost every
// point: below a window of +-5 standard deviations it is a member, above it is
// not, and the few hundred inside are listed in shared memory, where a
// histogram and a rank count find the last member.  The keys are never stored
// (one bit per point is).  When the window misses (about one unit in 10^6 at five
// standard deviations), an 8-bit radix select over four passes recomputes the keys.
// The window is narrower where the list would not hold it (libraries of about half
// of more than 2.6 million points), down to three standard deviations (one unit in
// 400 misses); where not even those fit, the pass is left out and the radix select
// is all there is.
//
// Bound: issue (the 64-bit multiplies of Philox are half of the instructions)
// and, for short manifolds, the latency between its barriers: five CTAs per SM
// (48 registers; the listed keys sized by N_m) hide more of it than three.
// Sweep of 4*10^5 libraries of N_m = 10^4: 13.9 ms with the scan's membership
// words (keys stored and four radix passes over them: 20.0 ms); 27000 of N_m =
// 4000: 0.52 ms (0.63); 10^4 of N_m = 10^5: 2.9 ms (26.4).
//
// Output: realizations that read a distance indexing table get one bit per
// position of the query order; the others their library as a list in query
// order, the order the neighbour search visits it in (spatially coherent
// runs).  The checking copy is compacted in ascending m.
#include <limits.h>

#include <algorithm>

#include "bits.cuh"
#include "ccm_internal.h"
#include "launch.cuh"

namespace ccm {
namespace {

// Philox4x64-10 (Salmon et al., SC'11): ten rounds, two 64x64->128 products per
// round, round keys bumped by the Weyl constants between rounds.  Writes the
// four output words.
__device__ __forceinline__ void philox_block(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                                             uint64_t k0, uint64_t k1, uint64_t (&w)[4]) {
  const uint64_t M0 = 0xD2E7470EE14C6C93ULL, M1 = 0xCA5A826395121157ULL;
  const uint64_t W0 = 0x9E3779B97F4A7C15ULL, W1 = 0xBB67AE8584CAA73BULL;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    if (round > 0) {
      k0 += W0;
      k1 += W1;
    }
    const unsigned __int128 p0 = (unsigned __int128)M0 * c0, p1 = (unsigned __int128)M1 * c2;
    const uint64_t hi0 = (uint64_t)(p0 >> 64), lo0 = (uint64_t)p0;
    const uint64_t hi1 = (uint64_t)(p1 >> 64), lo1 = (uint64_t)p1;
    const uint64_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  w[0] = c0;
  w[1] = c1;
  w[2] = c2;
  w[3] = c3;
}

// The Philox block holding the keys of points 8b .. 8b+7.
__device__ __forceinline__ void key_block(const UnitDesc& u, int b, uint64_t (&w)[4]) {
  const uint64_t c3 = ((uint64_t)u.j << 16) | ((uint64_t)u.E << 8) | (uint64_t)u.tau;
  philox_block((uint64_t)b, (uint64_t)u.k, (uint64_t)u.L, c3, u.seed, 0, w);
}

// 32-bit half number i (0..7) of a block: hi(w0), lo(w0), hi(w1), ..., lo(w3).
__device__ __forceinline__ uint32_t block_half(const uint64_t (&w)[4], int i) {
  const int q = i >> 1;
  const uint64_t x = (q == 0) ? w[0] : (q == 1) ? w[1] : (q == 2) ? w[2] : w[3];
  return (i & 1) ? (uint32_t)x : (uint32_t)(x >> 32);
}

// Stable compaction of the members among positions [0, n) by the whole block,
// warp by warp: warp w walks its contiguous segment 32 positions at a time
// (coalesced reads), counts members with a ballot, and after a block scan of
// the warp counts writes them in position order.  item(q) gives the manifold
// point at position q; is_member(m) decides membership.  `out` has room for
// `expect` entries: when the members number anything else (a sampler fault)
// nothing is compacted and out[0..expect) is filled with point 0 instead, so
// that later kernels reading the library stay in bounds.
template <typename Item, typename Member>
__device__ uint32_t block_compact(int n, Item item, Member is_member, int32_t* out,
                                  uint32_t expect, uint32_t* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  const int seg = ((n + nwarps - 1) / nwarps + 31) / 32 * 32;
  const int q0 = min(n, warp * seg), q1 = min(n, q0 + seg);
  uint32_t count = 0u;
  for (int q = q0 + lane; q - lane < q1; q += 32) {
    const bool mem = q < q1 && is_member(item(q));
    count += __popc(__ballot_sync(0xffffffffu, mem));
  }
  if (lane == 0) s_warp[warp] = count;
  __syncthreads();
  uint32_t base = 0u, total = 0u;
  for (int w = 0; w < nwarps; ++w) {
    base += (w < warp) ? s_warp[w] : 0u;
    total += s_warp[w];
  }
  __syncthreads();
  if (total != expect) {
    for (uint32_t q = threadIdx.x; q < expect; q += blockDim.x) out[q] = 0;
    return total;
  }
  for (int q = q0 + lane; q - lane < q1; q += 32) {
    const int m = q < q1 ? item(q) : 0;
    const bool mem = q < q1 && is_member(m);
    const unsigned bal = __ballot_sync(0xffffffffu, mem);
    if (mem) out[base + __popc(bal & ((1u << lane) - 1u))] = m;
    base += __popc(bal);
  }
  return total;
}

// The L-th smallest key of a unit whose window missed: an 8-bit radix select
// of its high half h* over four passes of recomputed keys, then the last of the
// points with that half that are taken (smallest m first).  Block-wide.
struct SelectScratch {
  uint32_t hist[256];
  uint32_t prefix, rank;
};
__device__ __noinline__ unsigned long long select_by_radix(const UnitDesc& u, SelectScratch& sc) {
  const int n_m = u.n_m, n_blocks = (n_m + 7) >> 3;
  const int lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    sc.prefix = 0u;
    sc.rank = (uint32_t)u.L;  // 1-based rank still to find within the current prefix
  }
  uint32_t mask = 0u;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    __syncthreads();
    for (int b = threadIdx.x; b < 256; b += blockDim.x) sc.hist[b] = 0u;
    __syncthreads();
    const uint32_t prefix = sc.prefix;
    for (int b = threadIdx.x; b < n_blocks; b += blockDim.x) {
      uint64_t w[4];
      key_block(u, b, w);
      for (int i = 0; i < 8; ++i) {
        const uint32_t h = block_half(w, i);
        if (8 * b + i < n_m && (h & mask) == prefix) atomicAdd(&sc.hist[(h >> shift) & 255u], 1u);
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      // the bin holding the rank: lane l sums bins 8l..8l+7, then a warp scan
      const uint32_t rank = sc.rank;
      uint32_t mine = 0u;
#pragma unroll
      for (int b = 0; b < 8; ++b) mine += sc.hist[lane * 8 + b];
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, incl >= rank);
      const int owner = __ffs(hit) - 1;  // exists: the histogram holds >= rank keys
      if (lane == owner) {
        uint32_t cum = incl - mine;
        int b = lane * 8;
        for (; b < lane * 8 + 7; ++b) {
          if (cum + sc.hist[b] >= rank) break;
          cum += sc.hist[b];
        }
        sc.prefix = prefix | ((uint32_t)b << shift);
        sc.rank = rank - cum;
      }
    }
    mask |= 255u << shift;
  }
  __syncthreads();
  const uint32_t hstar = sc.prefix;    // high half of the L-th smallest key
  const uint32_t take_ties = sc.rank;  // points with h == h* to take, smallest m first
  __syncthreads();
  // warp 0 finds the last tie taken (no shared state but the prefix word)
  if (threadIdx.x < 32) {
    uint32_t seen = 0u;
    int mtie = -1;
    for (int b0 = 0; b0 < n_blocks && mtie < 0; b0 += 32) {
      uint64_t w[4];
      key_block(u, min(b0 + lane, n_blocks - 1), w);
      uint32_t ties = 0u;
      for (int i = 0; i < 8; ++i)
        if (b0 + lane < n_blocks && 8 * (b0 + lane) + i < n_m && block_half(w, i) == hstar)
          ties |= 1u << i;
      uint32_t incl = __popc(ties);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, seen + incl >= take_ties);
      if (hit) {
        const int owner = __ffs(hit) - 1;
        uint32_t before = seen + incl - __popc(ties);
        for (uint32_t k = before + 1; k < take_ties; ++k) ties &= ties - 1u;  // drop earlier ties
        mtie = __shfl_sync(0xffffffffu, 8 * (b0 + lane) + __ffs(ties) - 1, owner);
      }
      seen += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) sc.prefix = (uint32_t)mtie;
  }
  __syncthreads();
  return ((unsigned long long)hstar << 32) | sc.prefix;
}

// Keys listed around the L-th smallest, at most: ten standard deviations of the
// rank (at most sqrt(n)/2) and as many again as they may spread.
__host__ __device__ constexpr int window_keys(int n) {
  int root = 1;
  while ((int64_t)root * root < n) root <<= 1;  // sqrt(n) to twice it
  return root * 6 + 96 < 8192 ? root * 6 + 96 : 8192;
}
constexpr int kBinKeys = 64;   // of them, keys of the bin that holds it

__global__ void __launch_bounds__(kSamplerThreads, 5)
sampler_kernel(SamplerParams p, int64_t first_unit, int window) {
  extern __shared__ __align__(16) unsigned long long s_win[];  // listed keys, then
  __shared__ unsigned long long s_bin_keys[kBinKeys], s_last;
  uint32_t* s_bits = reinterpret_cast<uint32_t*>(s_win + window);  // bit m: point m is a member
  __shared__ SelectScratch s_sel;
  __shared__ uint32_t s_warp[32];
  __shared__ uint32_t s_below, s_listed, s_rank, s_bin, s_in_bin, s_total;

  chain_begin();
  const int64_t uidx = first_unit + blockIdx.x;
  const UnitDesc u = p.units[uidx];
  const int n_m = u.n_m, L = u.L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (L < 1 || L > n_m) {
    if (tid == 0) atomicOr(p.err, kErrSampler);
    return;
  }
  const int n_blocks = (n_m + 7) >> 3, words = (n_m + 31) >> 5;
  // a manifold too long for the bits keeps only the last member's key
  const bool keep = n_m <= kSamplerBitsMax;
  unsigned char* bytes = reinterpret_cast<unsigned char*>(s_bits);

  // The window [lo, hi] of high halves: L/N_m of the range, +-5 standard
  // deviations of the rank (and a few keys more).
  const float pf = (float)L / (float)n_m, sd = sqrtf((float)L * fmaxf(1.f - pf, 0.f));
  const float half_keys = fminf(5.f * sd + 8.f, 0.45f * (float)window);
  const bool look = half_keys >= 3.f * sd;
  const uint64_t centre = ((uint64_t)L << 32) / (uint32_t)n_m;
  const uint64_t half = (uint64_t)(half_keys * (4294967296.f / (float)n_m));
  const uint32_t lo = centre > half ? (uint32_t)min(centre - half, (uint64_t)0xffffffffu) : 0u;
  const uint32_t hi = (uint32_t)min(centre + half, (uint64_t)0xffffffffu);
  for (int b = tid; b < 256; b += kSamplerThreads) s_sel.hist[b] = 0u;
  if (tid == 0) {
    s_below = s_listed = s_in_bin = s_total = 0u;
    s_rank = 0u;
    s_bin = 0xffffffffu;
    for (int b = n_blocks; b < 4 * words && keep; ++b) bytes[b] = 0;  // the last word's unused bytes
  }
  __syncthreads();
  uint32_t below = 0u;
  for (int b = tid; b < n_blocks && look; b += kSamplerThreads) {
    uint64_t w[4];
    key_block(u, b, w);
    uint32_t byte = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint32_t h = block_half(w, i);
      if (h < lo) byte |= 1u << i;
      if (h - lo <= hi - lo && 8 * b + i < n_m) {
        const uint32_t at = atomicAdd(&s_listed, 1u);
        if (at < (uint32_t)window) s_win[at] = ((unsigned long long)h << 32) | (uint32_t)(8 * b + i);
      }
    }
    if (8 * b + 8 > n_m) byte &= (1u << (n_m - 8 * b)) - 1u;
    below += __popc(byte);
    if (keep) bytes[b] = (unsigned char)byte;
  }
  below = __reduce_add_sync(0xffffffffu, below);
  if (lane == 0 && below) atomicAdd(&s_below, below);
  __syncthreads();
  const uint32_t listed = s_listed, sum_below = s_below;
  // members among the listed keys; 0 and all of them need no search
  const uint32_t want = (uint32_t)L - sum_below;
  bool found = look && (uint32_t)L >= sum_below && listed <= (uint32_t)window && want <= listed;
  if (found && want > 0u && want < listed) {
    // bins of equal width over the window: the one holding the last member,
    // then its rank among that bin's keys
    const uint64_t scale = (256ull << 24) / ((uint64_t)(hi - lo) + 1u);
    auto bin_of = [&](unsigned long long key) {
      return min(255u, (uint32_t)(((uint32_t)(key >> 32) - lo) * scale >> 24));
    };
    for (uint32_t q = tid; q < listed; q += kSamplerThreads) atomicAdd(&s_sel.hist[bin_of(s_win[q])], 1u);
    __syncthreads();
    if (tid < 32) {
      uint32_t mine = 0u;
#pragma unroll
      for (int b = 0; b < 8; ++b) mine += s_sel.hist[lane * 8 + b];
      uint32_t incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const unsigned hit = __ballot_sync(0xffffffffu, incl >= want);
      if (lane == __ffs(hit) - 1) {
        uint32_t cum = incl - mine;
        int b = lane * 8;
        for (; b < lane * 8 + 7; ++b) {
          if (cum + s_sel.hist[b] >= want) break;
          cum += s_sel.hist[b];
        }
        s_bin = (uint32_t)b;
        s_rank = want - cum;
      }
    }
    __syncthreads();
    for (uint32_t q = tid; q < listed; q += kSamplerThreads) {
      const unsigned long long key = s_win[q];
      if (bin_of(key) == s_bin) {
        const uint32_t at = atomicAdd(&s_in_bin, 1u);
        if (at < (uint32_t)kBinKeys) s_bin_keys[at] = key;
      }
    }
    __syncthreads();
    const uint32_t in_bin = s_in_bin;
    found = in_bin <= (uint32_t)kBinKeys;
    if (found && tid < (int)in_bin) {
      const unsigned long long key = s_bin_keys[tid];
      uint32_t less = 0u;
      for (uint32_t q = 0; q < in_bin; ++q) less += s_bin_keys[q] < key ? 1u : 0u;
      if (less + 1u == s_rank) s_last = key;
    }
    __syncthreads();
  }
  // the last member's key; the members are the points whose key is not above it
  const unsigned long long last = !found            ? select_by_radix(u, s_sel)
                                  : want == 0u      ? ((unsigned long long)lo << 32) - 1ull
                                  : want == listed ? ((unsigned long long)hi << 32) | 0xffffffffull
                                                    : s_last;
  if (keep && found) {
    for (uint32_t q = tid; q < listed; q += kSamplerThreads) {
      const unsigned long long key = s_win[q];
      if (key <= last) atomicOr(&s_bits[(uint32_t)key >> 5], 1u << ((uint32_t)key & 31u));
    }
  } else if (keep) {
    for (int b = tid; b < n_blocks; b += kSamplerThreads) {
      uint64_t w[4];
      key_block(u, b, w);
      uint32_t byte = 0u;
      for (int i = 0; i < 8; ++i) {
        const unsigned long long key = ((unsigned long long)block_half(w, i) << 32) | (uint32_t)(8 * b + i);
        if (8 * b + i < n_m && key <= last) byte |= 1u << i;
      }
      bytes[b] = (unsigned char)byte;
    }
  }
  __syncthreads();
  auto is_member = [&](int m) {
    if (keep) return ((s_bits[m >> 5] >> (m & 31)) & 1u) != 0u;
    uint64_t w[4];
    key_block(u, m >> 3, w);
    return (((unsigned long long)block_half(w, m & 7) << 32) | (uint32_t)m) <= last;
  };
  const int32_t* ord = p.order + u.order_off;
  uint32_t total = 0u;
  if (u.table_R > 0 && !p.list_all) {
    // one bit per position of the query order, eight words at a time per warp
    uint32_t* out = p.bits + u.bits_off;
    uint32_t count = 0u;
    for (int w0 = warp * 8; w0 < words; w0 += kSamplerThreads / 32 * 8) {
      uint32_t mine = 0u;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int pos = (w0 + i) * 32 + lane;
        const bool mem = pos < n_m && is_member(ord[min(pos, n_m - 1)]);
        const uint32_t word = __ballot_sync(0xffffffffu, mem);
        if (lane == i) mine = word;
      }
      if (lane < 8 && w0 + lane < words) out[w0 + lane] = mine;
      count += __popc(mine);
    }
    count = __reduce_add_sync(0xffffffffu, count);
    if (lane == 0) atomicAdd(&s_total, count);
    __syncthreads();
    total = s_total;
  } else {
    // the library in query order (the order the neighbour search visits it in)
    total = block_compact(n_m, [&](int q) { return ord[q]; }, is_member,
                          p.lib + u.lib_off, (uint32_t)L, s_warp);
  }
  if (total != (uint32_t)L) {  // not a permutation, or a lost tie: report, never guess
    if (tid == 0) atomicOr(p.err, kErrSampler);
    return;
  }
  if (p.dbg_lib) {  // checking copy in ascending m, once per target of this library
    for (int t = 0; t < u.n_targets; ++t) {
      __syncthreads();
      block_compact(n_m, [](int q) { return q; }, is_member,
                    p.dbg_lib + p.targets[u.tgt_off + t].lib_dbg_off, (uint32_t)L, s_warp);
    }
  }
}

}  // namespace

cudaError_t sampler_prepare() {
  return cudaFuncSetAttribute(sampler_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              kSamplerBitsMax / 8 + window_keys(INT_MAX) * 8);
}

cudaError_t launch_sampler(const SamplerParams& p, int64_t first_unit, int64_t count, int max_nm,
                           LaunchStream s) {
  const int window = p.window > 0 ? std::min(p.window, window_keys(max_nm)) : window_keys(max_nm);
  const size_t smem = (size_t)window * 8 + (size_t)((std::min(max_nm, kSamplerBitsMax) + 31) / 32) * 4;
  for (int64_t off = 0; off < count; off += 0x7fffffff) {
    const unsigned grid = (unsigned)std::min<int64_t>(count - off, 0x7fffffff);
    const cudaError_t e =
        launch_chained(sampler_kernel, dim3(grid), kSamplerThreads, smem, s, p, first_unit + off, window);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Membership words of the scan's realization groups: word pos of a group holds
// bit r when position pos of the query order is in the library of its r-th
// realization; the words past the last position are zero (the positions that
// pad a table row).  A warp turns 32 positions of 32 realizations at a time:
// lane r reads the realization's bits, the transpose leaves a word per position.
__global__ void __launch_bounds__(256) member_words_kernel(const UnitDesc* units,
                                                          const MemberGroup* groups,
                                                          const uint32_t* bits, uint32_t* words) {
  chain_begin();
  const MemberGroup g = groups[blockIdx.y];
  const UnitDesc& u = units[g.unit];
  const int n_m = u.n_m, per_unit = (n_m + 31) >> 5;
  const int lane = threadIdx.x & 31;
  const BitTranspose tr(lane);
  const uint32_t* src = bits + u.bits_off + (int64_t)min(lane, g.count - 1) * per_unit;
  uint32_t* dst = words + u.words_off;
  const int blocks = member_words(n_m) >> 5;
  // eight consecutive blocks a warp: the 32-byte sectors of `src` are used whole
  const int b0 = (blockIdx.x * 8 + (threadIdx.x >> 5)) * 8;
  for (int b = b0; b < min(b0 + 8, blocks); ++b) {
    const uint32_t w = (lane < g.count && b < per_unit) ? src[b] : 0u;
    dst[b * 32 + lane] = tr(w);
  }
}

cudaError_t launch_member_words(const UnitDesc* units, const MemberGroup* groups, int64_t n_groups,
                                int max_nm, const uint32_t* bits, uint32_t* words, LaunchStream s) {
  const unsigned gx = (unsigned)((member_words(max_nm) / 32 + 63) / 64);
  for (int64_t off = 0; off < n_groups; off += 65535) {
    const dim3 grid(gx, (unsigned)std::min<int64_t>(n_groups - off, 65535));
    const cudaError_t e =
        launch_chained(member_words_kernel, grid, 256, 0, s, units, groups + off, bits, words);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace ccm
