// Distance indexing table (paper Sect. 3.2: a table of the sorted distances of
// every point, built once, from which the E+1 nearest neighbours of any
// subsample are read off instead of re-sorting all distances for every
// subsample; Sect. 3.2 and Fig. 2 describe it as a second pipeline that feeds
// the CCM transform).
//
// For one (library variable, E, tau) the table holds, for every query
// position pos of the query order, the R nearest manifold points of the query
// m = order[pos] over the WHOLE manifold, m itself left out (no neighbour
// list holds it), sorted by (FP32 squared distance, index), the same key the
// brute-force selection uses.  For a realization whose library is a subset of
// the manifold, the first E+1 table entries that are library members (outside
// the exclusion window) are exactly its E+1 nearest library neighbours:
// restricting a total order to a subset keeps its order.
//
// Layout: row after row, table[table_off + pos*stride + r], an entry being the
// point's position in the query order (16 bits when every manifold of the plan
// has fewer than 65536 points, else 32; rows are padded to a multiple of 64
// with position n_m, which no library holds).  A warp that walks a row reads 32
// ranks with one access, and neighbouring points have neighbouring positions,
// so lookups by position are coherent.  A float array of the same layout holds
// each entry's distance (the square root the simplex weights take of the FP32
// squared distance, computed the same way), or pairs of it and the single
// target's value at the point, so that the scan reads what the prediction needs
// from the row.
//
// Build: one CTA per row (compiled once per E).
//  * The manifold's points lie in query order, 32 to a chunk with its bounding
//    box over all E coordinates, 32 chunks to a superchunk with its own
//    (table.cu).  A superchunk, then a chunk, whose box lies farther than the
//    row's threshold is skipped whole: the box bound is formed in the
//    distance's own rounding order, so it is at most every FP32 squared
//    distance in the box.
//  * The threshold is a key (squared distance, index) under which between R
//    and C points lie: the previous row's (of the same point as it is, else
//    scaled to the wanted count: rows of one CTA are consecutive in query order,
//    so their neighbourhoods are alike), else the k-th smallest distance of a
//    sample (one histogram).  When the collected count misses [R, C], histograms
//    of the distances between the two sides narrow it down by a factor of 1024
//    each; where more than fit tie, of their indices.  Every point at or below
//    it is collected, so the R smallest are among them.  A chunk whose box lies
//    at the tied distance itself is skipped when its smallest index is above the
//    threshold's: equal points lie in index order, so of a value that fills half
//    a series the first few chunks are read.
//  * The collected keys are sorted by 1024 bins of the distance's bit pattern
//    below the threshold (256 per octave in the two octaves that hold most keys
//    of a manifold, 64 below, so a bin holds a handful) and, within a bin, by
//    counting smaller keys; a crowded bin (ties) falls back to a
//    bitonic sort.
//
// Bound: issue (67 %, ncu, E = 3: collecting and ranking about half each) and,
// at E = 10, the latency of the points in L2.  With the query order and the
// target series' preparation: 80 tables of N = 10^4 (E = 1..10, rows of 130 to
// 1000) 24 ms; 8 of N = 10^5 (E = 3..6) 29 ms.  A warp per row, two passes over
// all N_m distances (a sample and one pass from N = 32768) and bitonic sorts
// took 62 and 187 ms.
#include <stdint.h>

#include "ccm_internal.h"
#include "launch.cuh"

namespace ccm {
namespace {

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kBins = 1024;
constexpr int kSampleShift = 17;   // sample bins: 64 per octave, 16 octaves
constexpr int kCrowded = 128;      // keys of a bin ranked by counting, at most
constexpr int kAttempts = 256;     // thresholds tried for a row (a few)
constexpr int kSegment = 64;       // superchunks whose chunks are listed at a time

// Collected keys of a row, at most: twice as many as wanted (half as many again
// for long rows, whose shared memory is the limit), and the count a threshold
// aims at.  Keys beyond the row are collected but not ranked.
__host__ __device__ constexpr int capacity(int R) {
  return R + (R <= 1024 ? R : R <= 2048 ? 1024 : R / 2) + 64;
}
__host__ __device__ constexpr int wanted(int R) { return R + (capacity(R) - R) * 2 / 5; }

size_t build_smem(int max_R, int max_nm) {
  const int chunks = (max_nm + 31) / 32, supers = (chunks + 31) / 32;
  const int listed = chunks < kSegment * 32 ? chunks : kSegment * 32;
  return (size_t)kBins * 4 + (size_t)capacity(max_R) * 8 +
         ((size_t)capacity(max_R) + supers + listed + 8) * 2;
}

template <int E>
struct Point {
  float x[E];
};

// What is known of a row's threshold once one missed.
struct RowSearch {
  uint32_t lo, hi, step;          // squared distances under which too few, too many lie
  int lo_m, hi_m, below, above;   // indices likewise, among ties; the counts at the two sides
  bool have_lo, have_hi, halved, ties;
};

template <int kThreads>
struct BlockState {
  uint32_t scan[kThreads / 32], top, found, crowd;
  int supers, chunks, count, equal;
  RowSearch row;
};

// Lower bound of the squared distances of q to box i of an array of `n` boxes.
template <int E>
__device__ __forceinline__ uint32_t box_bound(const Point<E>& q, const float* b, int n, int i) {
  float lb = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const float g = fmaxf(fmaxf(__fsub_rn(b[2 * e * n + i], q.x[e]),
                                __fsub_rn(q.x[e], b[(2 * e + 1) * n + i])), 0.f);
    lb = (e == 0) ? __fmul_rn(g, g) : __fmaf_rn(g, g, lb);
  }
  return __float_as_uint(lb);
}

// Exclusive scan of the bins in place; thread t holds bins [t*B, (t+1)*B).  With
// rank > 0 also sh.found = the bin holding that (1-based) rank; sh.crowd: the
// largest bin.  Block-wide, ends behind a barrier.
template <int kThreads>
__device__ __forceinline__ void scan(uint32_t* bins, BlockState<kThreads>& sh, uint32_t rank) {
  constexpr int kPer = kBins / kThreads, kWarps = kThreads / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t v[kPer], sum = 0u, most = 0u;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    v[i] = bins[tid * kPer + i];
    sum += v[i];
    most = max(most, v[i]);
  }
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(kFullMask, incl, o);
    if (lane >= o) incl += y;
  }
  most = __reduce_max_sync(kFullMask, most);
  if (lane == 31) sh.scan[warp] = incl;
  if (lane == 0 && most > (uint32_t)kCrowded) sh.crowd = 1u;
  __syncthreads();
  uint32_t before = incl - sum;
#pragma unroll
  for (int w = 0; w < kWarps; ++w) before += (w < warp) ? sh.scan[w] : 0u;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    bins[tid * kPer + i] = before;
    if (rank > before && rank <= before + v[i]) sh.found = (uint32_t)(tid * kPer + i);
    before += v[i];
  }
  __syncthreads();
}

// The points within squared distance `most` of query q at position pos (to the bit),
// into the bins, which are cleared first: with m_from < 0 by (bits - from) >> shift,
// those below `from` to bin 0; else those at `most` with index m_from .. m_to by
// (index - m_from) >> shift.  Block-wide, behind the closing barrier.
template <int E, int kThreads>
__device__ __forceinline__ void distance_histogram(const Point<E>& q, const TableJob& jb,
                                                   const float* points, const int32_t* order, int pos,
                                                   uint32_t most, uint32_t from, int m_from, int m_to,
                                                   int shift, uint32_t* bins) {
  constexpr int kWarps = kThreads / 32;
  const int n_m = jb.n_m, n_chunks = (n_m + 31) >> 5, n_super = (n_chunks + 31) >> 5;
  const float* pts = points + jb.pts_off;
  const float* box = points + jb.box_off;
  const float* sbox = points + jb.sbox_off;
  const int32_t* least = reinterpret_cast<const int32_t*>(points + jb.least_off);
  const int32_t* ord = order + jb.order_off;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = threadIdx.x; i < kBins; i += kThreads) bins[i] = 0u;
  __syncthreads();
  for (int sc = 0; sc < n_super; ++sc) {
    if (box_bound(q, sbox, n_super, sc) > most || (m_from >= 0 && least[n_super * 32 + sc] > m_to))
      continue;
    const int ch = sc * 32 + lane;
    // (a warp takes every kWarps-th chunk: few superchunks would not share out)
    const bool keep = ch < n_chunks && lane % kWarps == warp &&
                      box_bound(q, box, n_super * 32, min(ch, n_chunks - 1)) <= most &&
                      (m_from < 0 || least[ch] <= m_to);
    for (unsigned left = __ballot_sync(kFullMask, keep); left; left &= left - 1u) {
      const int x0 = (sc * 32 + __ffs(left) - 1) * 32, x = x0 + lane;
      const float* src = pts + (int64_t)x0 * E + lane;
      float diff = __fsub_rn(q.x[0], src[0]);
      float acc = __fmul_rn(diff, diff);
#pragma unroll
      for (int e = 1; e < E; ++e) {
        diff = __fsub_rn(q.x[e], src[e * 32]);
        acc = __fmaf_rn(diff, diff, acc);
      }
      const uint32_t bits = __float_as_uint(acc);
      if (x >= n_m || x == pos || bits > most) continue;
      if (m_from < 0) {
        atomicAdd(&bins[bits < from ? 0u : (bits - from) >> shift], 1u);
      } else if (bits == most) {
        const int m = ord[x];
        if (m >= m_from && m <= m_to) atomicAdd(&bins[(m - m_from) >> shift], 1u);
      }
    }
    __syncwarp();
  }
  __syncthreads();
}

// A row's next threshold after (tb, tm) missed: `c` points lie at or below it, `equal`
// at tb itself (whatever their index).  Block-wide, behind the closing barrier; in
// sh.row what is known of the row (`first`: nothing yet).  Not inlined: few rows come
// here, and its registers are the collecting loop's.
struct Threshold {
  uint32_t tb, tm;
};
template <int E, int kThreads>
__device__ __noinline__ Threshold next_threshold(const Point<E> q, const TableJob* jobs,
                                                 const float* points, const int32_t* order, int pos,
                                                 Threshold t, int c, int equal, bool first,
                                                 uint32_t* bins, BlockState<kThreads>* state) {
  BlockState<kThreads>& sh = *state;
  const TableJob& jb = jobs[blockIdx.y];
  const int n_m = jb.n_m, R = jb.R, C = capacity(R), target = wanted(R);
  RowSearch s = {0u, 0u, 1u << 19, -1, 0, 0, 0, false, false, false, false};
  if (!first) s = sh.row;
  __syncthreads();  // read by all before it is written
  bool tied = false;  // just now: an index is guessed first
  if (s.ties) {
    if (c < R) {
      s.lo_m = (int)t.tm;
      s.below = c;
    } else {
      s.hi_m = (int)t.tm;
      s.above = c;
    }
  } else {
    // a tie that does not fit, known at once (when no tie was left out: a
    // carried-over threshold may have an index)
    tied = t.tm == 0xffffffffu && c > C && c - equal < R;
    if (c < R) {
      s.lo = t.tb;
      s.have_lo = true;
      s.below = c;
    } else {
      s.hi = t.tb;
      s.have_hi = true;
      s.above = c;
    }
    t.tm = 0xffffffffu;
    if (tied) s.below = c - equal;
  }
  const bool step = !s.ties && !tied && (!(s.have_lo && s.have_hi) || !s.halved);
  if (step) {  // (of distances that differ, a step or the middle of two mostly holds)
    if (s.step < (1u << 30)) s.step <<= 1;
    s.halved = s.have_lo && s.have_hi;
    if (s.halved) t.tb = s.lo + (s.hi - s.lo) / 2u;
    else if (s.have_lo) t.tb = s.lo > 0xffffffffu - s.step ? 0xffffffffu : s.lo + s.step;
    else t.tb = s.hi > s.step ? s.hi - s.step : 0u;
  }
  // (four turns cover 32 bits; the bound ends the loop whatever the counts say)
  for (int turn = 0; !step && !tied && turn < 8; ++turn) {
    const uint32_t from = s.have_lo ? s.lo + 1u : 0u;
    const uint32_t span = s.ties ? (uint32_t)(s.hi_m - s.lo_m - 1) : s.hi - from;
    int shift = 0;
    while (span >> shift >= (uint32_t)kBins) ++shift;
    const int known = s.ties ? s.below : 0;
    distance_histogram<E, kThreads>(q, jb, points, order, pos, s.ties ? t.tb : s.hi, from,
                                    s.ties ? s.lo_m + 1 : -1, s.hi_m, shift, bins);
    scan<kThreads>(bins, sh, (uint32_t)(target - known));
    // the bin in which the wanted count is reached; the counts before it and through it
    const uint32_t f = sh.found;
    int before = (int)bins[f] + known;
    const int through = f + 1u < (uint32_t)kBins ? (int)bins[f + 1u] + known : s.above;
    __syncthreads();
    if (f == 0u) before = s.below;  // by distance, the first bin holds what lies below `from`, too
    // the last key of the bin before, and of this one
    const uint32_t lowest = s.ties ? (uint32_t)(s.lo_m + 1) : from;
    const uint32_t was = lowest + (f << shift) - 1u;
    const uint32_t end = lowest + (uint32_t)min((uint64_t)span, ((uint64_t)(f + 1u) << shift) - 1u);
    if (through <= C || before >= R) {
      const uint32_t key = through <= C ? end : was;
      if (s.ties) t.tm = key;
      else t.tb = key;
      break;
    }
    s.below = before;
    s.above = through;
    if (s.ties) {
      s.lo_m = (int)was;
      s.hi_m = (int)end;
    } else {
      if (f > 0u) {
        s.lo = was;
        s.have_lo = true;
      }
      s.hi = end;
      tied = shift == 0;  // one distance is left
    }
  }
  if (tied) {
    // more than fit tie at hi: up to an index, first guessed as if the tied points'
    // were spread evenly
    s.ties = true;
    s.lo_m = -1;
    s.hi_m = n_m - 1;
    t.tb = s.hi;
    t.tm = (uint32_t)((int64_t)n_m * (target - s.below) / (s.above - s.below));
  }
  if (threadIdx.x == 0) sh.row = s;
  __syncthreads();
  return t;
}

// (nine CTAs of 128 threads an SM for E <= 6: eight take 7 to 13 % longer)
template <int E, int kThreads>
__global__ void __launch_bounds__(kThreads, (E <= 6 ? 1152 : 1024) / kThreads)
table_build_kernel(const float* series, const TableJob* jobs, const float* points,
                   const int32_t* order, const int32_t* inverse, void* table, float* table_dist,
                   int pairs, int u16, int rows_per_cta, int cap, int32_t* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ BlockState<kThreads> sh;
  constexpr int kWarps = kThreads / 32;
  chain_begin();
  const TableJob jb = jobs[blockIdx.y];
  const int n_m = jb.n_m, R = jb.R, C = capacity(R);
  const int row0 = blockIdx.x * rows_per_cta;
  if (jb.E != E || row0 >= n_m) return;  // the same for the whole CTA
  const int row1 = min(n_m, row0 + rows_per_cta);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned below_lane = (1u << lane) - 1u;
  const int n_chunks = (n_m + 31) >> 5, n_super = (n_chunks + 31) >> 5;
  uint32_t* s_bin = reinterpret_cast<uint32_t*>(smem);                   // [kBins]
  uint32_t* s_bits = s_bin + kBins;                                      // [cap]
  uint32_t* s_m = s_bits + cap;                                          // [cap]
  uint16_t* s_idx = reinterpret_cast<uint16_t*>(s_m + cap);              // [cap]
  uint16_t* s_super = s_idx + cap;                                       // [n_super]
  uint16_t* s_chunk = s_super + n_super;
  const float* pts = points + jb.pts_off;          // [chunk][E][32]
  const float* box = points + jb.box_off;          // [2E][n_super*32]
  const float* sbox = points + jb.sbox_off;        // [2E][n_super]
  const int32_t* least = reinterpret_cast<const int32_t*>(points + jb.least_off);  // [n_super*32]
  const int32_t* sleast = least + n_super * 32;    // [n_super]
  const int32_t* ord = order + jb.order_off;
  const int32_t* inv = inverse + jb.order_off;
  const int off = (E - 1) * jb.tau;
  const bool has_value = pairs && jb.tv_i >= 0;
  const float* tv = series + jb.series_off + (int64_t)(jb.tv_i >= 0 ? jb.tv_i : 0) * jb.n + off;

  Point<E> q;
  auto bound = [&](const float* b, int n, int i) { return box_bound(q, b, n, i); };
  auto scan_bins = [&](uint32_t rank) { scan<kThreads>(s_bin, sh, rank); };
  constexpr int kPer = kBins / kThreads;
  auto clear_bins = [&]() {
#pragma unroll
    for (int i = 0; i < kPer; ++i) s_bin[tid + i * kThreads] = 0u;
  };

  const int target = wanted(R);
  const int stride = jb.sample;            // the sample: every stride-th point,
  const int n_sample = n_m / stride;       // [E][n_sample]
  const float* smp = points + jb.sample_off;
  uint32_t tb = 0xffffffffu, tm = 0xffffffffu;  // the threshold
  bool guess = false;  // tb, tm are carried over from the previous row
  int distrust = 0;    // rows left that sample at once: a carried threshold missed
  uint32_t kept_tb = tb;  // the previous row's threshold itself (its tm is tm)

  for (int pos = row0; pos < row1; ++pos) {
    bool same = pos > row0;  // the previous row's point again: its threshold fits
    {
      const float* c = pts + (int64_t)(pos >> 5) * (E * 32) + (pos & 31);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const float x = c[e * 32];
        same = same && x == q.x[e];
        q.x[e] = x;
      }
    }
    bool all = n_m - 1 <= C;  // everything fits: no threshold
    bool sampled = false, missed = false;
    if (all) tb = tm = 0xffffffffu;
    if (same && !all) {
      tb = kept_tb;
      guess = true;
    }
    int c = 0;
    for (int attempt = 0;; ++attempt) {
      if (!all && !guess && !sampled) {
        // the k-th smallest sampled distance, to a bin
        sampled = true;
        if (tid == 0) sh.top = 0u;
        __syncthreads();
        uint32_t top = 0u;  // the farthest any point can be
        for (int i = tid; i < n_super; i += kThreads) {
          float ub = 0.f;
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const float g = fmaxf(fabsf(__fsub_rn(sbox[2 * e * n_super + i], q.x[e])),
                                  fabsf(__fsub_rn(q.x[e], sbox[(2 * e + 1) * n_super + i])));
            ub = __fmaf_rn(g, g, ub);
          }
          top = max(top, __float_as_uint(ub));
        }
        top = __reduce_max_sync(kFullMask, top);
        if (lane == 0) atomicMax(&sh.top, top);
        __syncthreads();
        // 16 octaves up to the farthest point; where the k-th lies below them, all
        // that is below in coarser bins, the first of which stands for distance 0
        top = sh.top + (1u << 21);
        uint32_t base = top > (uint32_t)kBins << kSampleShift ? top - ((uint32_t)kBins << kSampleShift) : 0u;
        for (int shift = kSampleShift;;) {
          clear_bins();
          if (tid == 0) sh.found = kBins;
          __syncthreads();
          for (int i = tid; i < n_sample; i += kThreads) {
            float diff = __fsub_rn(q.x[0], smp[i]);
            float acc = __fmul_rn(diff, diff);
#pragma unroll
            for (int e = 1; e < E; ++e) {
              diff = __fsub_rn(q.x[e], smp[e * n_sample + i]);
              acc = __fmaf_rn(diff, diff, acc);
            }
            const uint32_t bits = __float_as_uint(acc);
            if (bits < top)
              atomicAdd(&s_bin[bits < base ? 0u : min((bits - base) >> shift, (uint32_t)kBins - 1u)], 1u);
          }
          __syncthreads();
          scan_bins(stride == 1 ? (uint32_t)R + 1u : (uint32_t)((target + stride - 1) / stride + 1));
          const uint32_t found = sh.found;
          __syncthreads();  // read by all before it is reset
          if (found == 0u && base > 0u) {
            top = base + (1u << kSampleShift);
            base = 0u;
            while ((top - 1u) >> shift >= (uint32_t)kBins) ++shift;
            continue;
          }
          tb = found == (uint32_t)kBins ? 0xffffffffu : found == 0u ? 0u : base + ((found + 1u) << shift) - 1u;
          break;
        }
        tm = 0xffffffffu;
      }
      // collect every point at or below the threshold
      const bool limited = tm != 0xffffffffu;
      auto reaches = [&](uint32_t b, const int32_t* smallest, int i) {
        bool yes = b <= tb;
        if (limited && b == tb) yes = (uint32_t)smallest[i] <= tm;
        return yes;
      };
      __syncthreads();
      if (tid == 0) sh.supers = sh.count = sh.equal = 0;
      __syncthreads();
      for (int i = tid; i < n_super; i += kThreads)
        if (reaches(bound(sbox, n_super, i), sleast, i)) s_super[atomicAdd(&sh.supers, 1)] = (uint16_t)i;
      __syncthreads();
      const int supers = sh.supers;
      int equal = 0;
      for (int g0 = 0; g0 < supers; g0 += kSegment) {
        if (g0 > 0) __syncthreads();  // the previous segment's list has been read
        if (tid == 0) sh.chunks = 0;
        __syncthreads();
        for (int i = g0 + warp; i < min(supers, g0 + kSegment); i += kWarps) {
          const int ch = s_super[i] * 32 + lane;
          const bool keep = ch < n_chunks && reaches(bound(box, n_super * 32, min(ch, n_chunks - 1)), least, ch);
          const unsigned bal = __ballot_sync(kFullMask, keep);
          int at = 0;
          if (lane == 0 && bal) at = atomicAdd(&sh.chunks, __popc(bal));
          at = __shfl_sync(kFullMask, at, 0);
          if (keep) s_chunk[at + __popc(bal & below_lane)] = (uint16_t)ch;
        }
        __syncthreads();
        const int chunks = sh.chunks;
        auto collect = [&](int x, uint32_t bits, uint32_t m) {  // position x (past the end: not valid)
          bool hit = x < n_m && x != pos && bits <= tb;
          unsigned bal = __ballot_sync(kFullMask, hit);
          if (bal == 0u) return;
          const unsigned eq = __ballot_sync(kFullMask, hit && bits == tb);
          if (eq != 0u) {  // ties with the threshold: up to index tm
            equal += __popc(eq);
            hit = hit && (bits < tb || m <= tm);
            bal = __ballot_sync(kFullMask, hit);
          }
          int at = 0;
          if (lane == 0) at = atomicAdd(&sh.count, __popc(bal));
          at = __shfl_sync(kFullMask, at, 0) + __popc(bal & below_lane);
          if (hit && at < C) {
            s_bits[at] = bits;
            s_m[at] = m;
          }
        };
        // kAhead chunks' points are on their way while one is compared
        constexpr int kAhead = E <= 4 ? 4 : E <= 6 ? 3 : 2;
        float c[kAhead][E];
        int mm[kAhead];
        auto load = [&](int i, float (&f)[E], int& m) {
          const int ch = s_chunk[min(i, chunks - 1)];
          const float* src = pts + (int64_t)ch * (E * 32) + lane;
#pragma unroll
          for (int e = 0; e < E; ++e) f[e] = src[e * 32];
          m = __ldg(ord + min(ch * 32 + lane, n_m - 1));
        };
        if (warp < chunks) {
#pragma unroll
          for (int d = 0; d < kAhead; ++d) load(warp + d * kWarps, c[d], mm[d]);
        }
        for (int i0 = warp; i0 < chunks; i0 += kAhead * kWarps) {
#pragma unroll
          for (int d = 0; d < kAhead; ++d) {
            const int i = i0 + d * kWarps;
            if (i >= chunks) break;
            float diff = __fsub_rn(q.x[0], c[d][0]);
            float acc = __fmul_rn(diff, diff);
#pragma unroll
            for (int e = 1; e < E; ++e) {
              diff = __fsub_rn(q.x[e], c[d][e]);
              acc = __fmaf_rn(diff, diff, acc);
            }
            const int m = mm[d];
            if (i + kAhead * kWarps < chunks) load(i + kAhead * kWarps, c[d], mm[d]);
            collect(s_chunk[i] * 32 + lane, __float_as_uint(acc), (uint32_t)m);
          }
        }
      }
      if (lane == 0 && equal) atomicAdd(&sh.equal, equal);
      __syncthreads();
      c = sh.count;
      if (c >= R && c <= C) break;
      if (attempt == kAttempts) {  // never: the bisection has ended before
        if (tid == 0) atomicOr(err, kErrTable);
        c = min(c, C);
        break;
      }
      const int equal_all = sh.equal;
      if (guess && !(tm == 0xffffffffu && c > C && c - equal_all < R)) {
        // the carried threshold missed (and shows no tie): sample, here and for some rows
        guess = false;
        distrust = 6;
        continue;
      }
      guess = false;
      sampled = true;
      const Threshold next = next_threshold<E, kThreads>(q, jobs, points, order, pos, Threshold{tb, tm},
                                                         c, equal_all, !missed, s_bin, &sh);
      tb = next.tb;
      tm = next.tm;
      missed = true;
    }
    const int kept = min(R, c);

    // sort: count, scan, scatter by bin (ascending distance), rank inside bins
    clear_bins();
    if (tid == 0) sh.crowd = sh.top = 0u;
    __syncthreads();
    uint32_t top = tb;
    if (all) {  // no threshold: bins below the largest distance
      top = 0u;
      for (int t = tid; t < c; t += kThreads) top = max(top, s_bits[t]);
      top = __reduce_max_sync(kFullMask, top);
      if (lane == 0) atomicMax(&sh.top, top);
      __syncthreads();
      top = sh.top;
    }
    auto bin_of = [&](uint32_t bits) {
      const uint32_t d = top - bits;  // 2^23 bit patterns an octave
      const uint32_t b = d < 2u << 23 ? d >> 15 : min(512u + ((d - (2u << 23)) >> 17), (uint32_t)kBins - 1u);
      return (uint32_t)kBins - 1u - b;
    };
    for (int t = tid; t < c; t += kThreads) atomicAdd(&s_bin[bin_of(s_bits[t])], 1u);
    __syncthreads();
    scan_bins(0u);
    const int64_t base = jb.table_off + (int64_t)pos * jb.stride;
    // each entry's distance (the epilogue's square root), beside it; with pairs,
    // together with the target's value at the entry's point (what the
    // prediction weighs; 0 in a table without a target)
    auto emit = [&](int rank, uint32_t bits, float value, int at) {
      const float d = sqrt_hw(__uint_as_float(bits));
      if (pairs)
        reinterpret_cast<float2*>(table_dist)[base + rank] = make_float2(d, value);
      else
        table_dist[base + rank] = d;
      if (u16) static_cast<uint16_t*>(table)[base + rank] = (uint16_t)at;
      else static_cast<int32_t*>(table)[base + rank] = at;
    };
    if (sh.crowd == 0u) {
      for (int t = tid; t < c; t += kThreads)
        s_idx[atomicAdd(&s_bin[bin_of(s_bits[t])], 1u)] = (uint16_t)t;
      __syncthreads();  // s_bin[b] is now the end of bin b
      for (int i = tid; i < c; i += kThreads) {
        const int t = s_idx[i];
        const uint32_t bits = s_bits[t], m = s_m[t];
        const uint32_t b = bin_of(bits);
        const int b0 = b > 0u ? (int)s_bin[b - 1u] : 0, b1 = (int)s_bin[b];
        int rank = b0;
        if (b0 >= R) continue;  // beyond the row
        const float value = has_value ? __ldg(tv + m) : 0.f;  // on their way while it is ranked
        const int at = __ldg(inv + m);
        for (int j = b0; j < b1; ++j) {
          const int o = s_idx[j];
          const uint32_t ob = s_bits[o];
          rank += (ob < bits || (ob == bits && s_m[o] < m)) ? 1 : 0;
        }
        if (rank < R) emit(rank, bits, value, at);
      }
    } else {
      // ascending-only bitonic network (mirrored first steps; positions at or
      // above c never take part)
      int n2 = 1;
      while (n2 < c) n2 <<= 1;
      for (int size = 2; size <= n2; size <<= 1) {
        for (int jj = size >> 1; jj > 0; jj >>= 1) {
          const bool mirror = jj == size >> 1;
          for (int t = tid; t < n2 >> 1; t += kThreads) {
            const int o = t & (jj - 1), a = 2 * t - o;
            const int b = mirror ? a - 2 * o + 2 * jj - 1 : a + jj;
            if (b < c) {
              const uint32_t ba = s_bits[a], bb = s_bits[b], ma = s_m[a], mb = s_m[b];
              if (bb < ba || (bb == ba && mb < ma)) {
                s_bits[a] = bb;
                s_bits[b] = ba;
                s_m[a] = mb;
                s_m[b] = ma;
              }
            }
          }
          __syncthreads();
        }
      }
      for (int r = tid; r < kept; r += kThreads)
        emit(r, s_bits[r], has_value ? __ldg(tv + s_m[r]) : 0.f, __ldg(inv + s_m[r]));
    }
    for (int r = kept + tid; r < jb.stride; r += kThreads) {
      if (u16) static_cast<uint16_t*>(table)[base + r] = (uint16_t)n_m;
      else static_cast<int32_t*>(table)[base + r] = n_m;
    }
    // the next row's threshold: this one's, moved towards the wanted count (the
    // exponent of a neighbourhood of two to three dimensions)
    guess = !all && distrust == 0;
    distrust -= distrust > 0 ? 1 : 0;
    kept_tb = tb;
    if (tm == 0xffffffffu && tb < 0x7f000000u) {
      const float f = __powf((float)target / (float)c, 0.8f);
      tb = __float_as_uint(__fmul_rn(__uint_as_float(tb), fminf(fmaxf(f, 0.5f), 2.f)));
    }
  }
}

}  // namespace

template <int E>
cudaError_t TableKernels<E>::prepare() {
  for (const auto fn : {table_build_kernel<E, 128>, table_build_kernel<E, 256>}) {
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)build_smem(kTableMaxR, kTableMaxNm));
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template <int E>
cudaError_t TableKernels<E>::launch(const float* series, const TableJob* jobs, int64_t n_jobs,
                                    int64_t n_rows, int max_nm, int max_R, const float* points,
                                    const int32_t* order, const int32_t* inverse, void* table,
                                    float* table_dist, int pairs, int u16, int32_t* err,
                                    LaunchStream s) {
  // consecutive rows share a CTA (and the threshold) once there are more rows
  // than fill the SMs twice
  const int64_t rows = n_rows / (2 * kSms * 8);
  const int per = (int)(rows < 1 ? 1 : rows > 32 ? 32 : rows);
  const size_t smem = build_smem(max_R, max_nm);
  const dim3 grid((unsigned)((max_nm + per - 1) / per), (unsigned)n_jobs);
  const int threads = max_R <= 1024 ? 128 : 256;
  return launch_chained(threads == 128 ? table_build_kernel<E, 128> : table_build_kernel<E, 256>, grid,
                        threads, smem, s, series, jobs, points, order, inverse, table, table_dist,
                        pairs, u16, per, capacity(max_R), err);
}

template struct TableKernels<CCM_E>;

}  // namespace ccm
