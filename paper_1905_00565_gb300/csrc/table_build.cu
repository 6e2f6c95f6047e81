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
//    and C points lie: the previous row's, scaled to the wanted count (rows of
//    one CTA are consecutive in query order, so their neighbourhoods are
//    alike), else the k-th smallest distance of a sample (one histogram); when
//    the collected count misses [R, C] it is bisected, over the index among
//    ties.  Every point at or below it is collected, so the R smallest are
//    among them.
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
constexpr int kAttempts = 256;     // thresholds tried for a row (a few; bisection needs 64)
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

template <int E, int kThreads>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads)
table_build_kernel(const float* series, const TableJob* jobs, const float* points,
                   const int32_t* order, const int32_t* inverse, void* table, float* table_dist,
                   int pairs, int u16, int rows_per_cta, int cap, int32_t* err) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t s_scan[kThreads / 32], s_top, s_found, s_crowd;
  __shared__ int s_supers, s_chunks, s_count, s_equal;
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
  const int32_t* ord = order + jb.order_off;
  const int32_t* inv = inverse + jb.order_off;
  const int off = (E - 1) * jb.tau;
  const bool has_value = pairs && jb.tv_i >= 0;
  const float* tv = series + jb.series_off + (int64_t)(jb.tv_i >= 0 ? jb.tv_i : 0) * jb.n + off;

  float q[E];
  // lower bound of the squared distances to box i of an array of `n` boxes
  auto bound = [&](const float* b, int n, int i) {
    float lb = 0.f;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const float g = fmaxf(fmaxf(__fsub_rn(b[2 * e * n + i], q[e]),
                                  __fsub_rn(q[e], b[(2 * e + 1) * n + i])), 0.f);
      lb = (e == 0) ? __fmul_rn(g, g) : __fmaf_rn(g, g, lb);
    }
    return __float_as_uint(lb);
  };
  // Exclusive scan of s_bin in place; thread t holds bins [t*B, (t+1)*B).  With
  // rank > 0 also s_found = the bin holding that (1-based) rank; s_crowd: the
  // largest bin.  Block-wide, ends behind a barrier.
  constexpr int kPer = kBins / kThreads;
  auto scan_bins = [&](uint32_t rank) {
    uint32_t v[kPer], sum = 0u, most = 0u;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      v[i] = s_bin[tid * kPer + i];
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
    if (lane == 31) s_scan[warp] = incl;
    if (lane == 0 && most > (uint32_t)kCrowded) s_crowd = 1u;
    __syncthreads();
    uint32_t before = incl - sum;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) before += (w < warp) ? s_scan[w] : 0u;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      s_bin[tid * kPer + i] = before;
      if (rank > before && rank <= before + v[i]) s_found = (uint32_t)(tid * kPer + i);
      before += v[i];
    }
    __syncthreads();
  };
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

  for (int pos = row0; pos < row1; ++pos) {
    {
      const float* c = pts + (int64_t)(pos >> 5) * (E * 32) + (pos & 31);
#pragma unroll
      for (int e = 0; e < E; ++e) q[e] = c[e * 32];
    }
    bool all = n_m - 1 <= C;  // everything fits: no threshold
    bool sampled = false, have_lo = false, have_hi = false, ties = false;
    uint32_t lo = 0u, hi = 0u, step = 1u << 19;
    int64_t lo_m = -1, hi_m = 0;
    if (all) tb = tm = 0xffffffffu;
    int c = 0;
    for (int attempt = 0;; ++attempt) {
      if (!all && !guess && !sampled) {
        // the k-th smallest sampled distance, to a bin
        sampled = true;
        if (tid == 0) s_top = 0u;
        __syncthreads();
        uint32_t top = 0u;  // the farthest any point can be
        for (int i = tid; i < n_super; i += kThreads) {
          float ub = 0.f;
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const float g = fmaxf(fabsf(__fsub_rn(sbox[2 * e * n_super + i], q[e])),
                                  fabsf(__fsub_rn(q[e], sbox[(2 * e + 1) * n_super + i])));
            ub = __fmaf_rn(g, g, ub);
          }
          top = max(top, __float_as_uint(ub));
        }
        top = __reduce_max_sync(kFullMask, top);
        if (lane == 0) atomicMax(&s_top, top);
        __syncthreads();
        // 16 octaves up to the farthest point; while the k-th lies below them,
        // the next 16 octaves down
        constexpr uint32_t kSpan = (uint32_t)kBins << kSampleShift;
        top = s_top + (1u << 21);
        for (;;) {
          const uint32_t base = top > kSpan ? top - kSpan : 0u;
          clear_bins();
          if (tid == 0) s_found = kBins;
          __syncthreads();
          for (int i = tid; i < n_sample; i += kThreads) {
            float diff = __fsub_rn(q[0], smp[i]);
            float acc = __fmul_rn(diff, diff);
#pragma unroll
            for (int e = 1; e < E; ++e) {
              diff = __fsub_rn(q[e], smp[e * n_sample + i]);
              acc = __fmaf_rn(diff, diff, acc);
            }
            const uint32_t bits = __float_as_uint(acc);
            if (bits < top)
              atomicAdd(&s_bin[bits < base ? 0u : min((bits - base) >> kSampleShift, (uint32_t)kBins - 1u)], 1u);
          }
          __syncthreads();
          scan_bins(stride == 1 ? (uint32_t)R + 1u : (uint32_t)((target + stride - 1) / stride + 1));
          const uint32_t found = s_found;
          __syncthreads();  // read by all before it is reset
          if (found == 0u && base > 0u) {
            top = base + (1u << kSampleShift);
            continue;
          }
          tb = found == (uint32_t)kBins ? 0xffffffffu : base + ((found + 1u) << kSampleShift) - 1u;
          break;
        }
        tm = 0xffffffffu;
      }
      // collect every point at or below the threshold
      __syncthreads();
      if (tid == 0) s_supers = s_count = s_equal = 0;
      __syncthreads();
      for (int i = tid; i < n_super; i += kThreads)
        if (bound(sbox, n_super, i) <= tb) s_super[atomicAdd(&s_supers, 1)] = (uint16_t)i;
      __syncthreads();
      const int supers = s_supers;
      int equal = 0;
      for (int g0 = 0; g0 < supers; g0 += kSegment) {
        if (g0 > 0) __syncthreads();  // the previous segment's list has been read
        if (tid == 0) s_chunks = 0;
        __syncthreads();
        for (int i = g0 + warp; i < min(supers, g0 + kSegment); i += kWarps) {
          const int ch = s_super[i] * 32 + lane;
          const bool keep = ch < n_chunks && bound(box, n_super * 32, min(ch, n_chunks - 1)) <= tb;
          const unsigned bal = __ballot_sync(kFullMask, keep);
          int at = 0;
          if (lane == 0 && bal) at = atomicAdd(&s_chunks, __popc(bal));
          at = __shfl_sync(kFullMask, at, 0);
          if (keep) s_chunk[at + __popc(bal & below_lane)] = (uint16_t)ch;
        }
        __syncthreads();
        const int chunks = s_chunks;
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
          if (lane == 0) at = atomicAdd(&s_count, __popc(bal));
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
            float diff = __fsub_rn(q[0], c[d][0]);
            float acc = __fmul_rn(diff, diff);
#pragma unroll
            for (int e = 1; e < E; ++e) {
              diff = __fsub_rn(q[e], c[d][e]);
              acc = __fmaf_rn(diff, diff, acc);
            }
            const int m = mm[d];
            if (i + kAhead * kWarps < chunks) load(i + kAhead * kWarps, c[d], mm[d]);
            collect(s_chunk[i] * 32 + lane, __float_as_uint(acc), (uint32_t)m);
          }
        }
      }
      if (lane == 0 && equal) atomicAdd(&s_equal, equal);
      __syncthreads();
      c = s_count;
      if (c >= R && c <= C) break;
      if (attempt == kAttempts) {  // never: the bisection has ended before
        if (tid == 0) atomicOr(err, kErrTable);
        c = min(c, C);
        break;
      }
      // missed: bracket the threshold
      if (ties) {
        if (c < R) lo_m = tm;
        else hi_m = tm;
        tm = (uint32_t)((lo_m + hi_m) >> 1);
        continue;
      }
      if (c < R) {
        lo = tb;
        have_lo = true;
      } else {
        hi = tb;
        have_hi = true;
        // points nearer than tb (known when no tie was left out: a carried-over
        // threshold may have an index)
        const int less = c - s_equal;
        if (tm == 0xffffffffu && less < R) {  // more than fit tie at tb: the smallest indices
          ties = true;
          hi_m = min((int64_t)tm, (int64_t)n_m);
          const int64_t want = (int64_t)(R + C) / 2 - less;
          tm = (uint32_t)min(hi_m - 1, (int64_t)n_m * want / (c - less));
          guess = false;
          sampled = true;
          continue;
        }
      }
      tm = 0xffffffffu;
      if (guess) {  // the carried threshold missed: sample, here and for some rows
        guess = false;
        distrust = 6;
        have_lo = have_hi = false;
        continue;
      }
      if (step < (1u << 30)) step <<= 1;
      if (have_lo && have_hi) tb = lo + (hi - lo) / 2u;
      else if (have_lo) tb = lo > 0xffffffffu - step ? 0xffffffffu : lo + step;
      else tb = hi > step ? hi - step : 0u;
    }

    // sort: count, scan, scatter by bin (ascending distance), rank inside bins
    clear_bins();
    if (tid == 0) s_crowd = s_top = 0u;
    __syncthreads();
    uint32_t top = tb;
    if (all) {  // no threshold: bins below the largest distance
      top = 0u;
      for (int t = tid; t < c; t += kThreads) top = max(top, s_bits[t]);
      top = __reduce_max_sync(kFullMask, top);
      if (lane == 0) atomicMax(&s_top, top);
      __syncthreads();
      top = s_top;
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
    if (s_crowd == 0u) {
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
      for (int r = tid; r < R; r += kThreads)
        emit(r, s_bits[r], has_value ? __ldg(tv + s_m[r]) : 0.f, __ldg(inv + s_m[r]));
    }
    for (int r = R + tid; r < jb.stride; r += kThreads) {
      if (u16) static_cast<uint16_t*>(table)[base + r] = (uint16_t)n_m;
      else static_cast<int32_t*>(table)[base + r] = n_m;
    }
    // the next row's threshold: this one's, moved towards the wanted count (the
    // exponent of a neighbourhood of two to three dimensions)
    guess = !all && distrust == 0;
    distrust -= distrust > 0 ? 1 : 0;
    if (!ties && tb < 0x7f000000u) {
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
  const int64_t rows = n_rows / (2 * 152 * 8);
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
