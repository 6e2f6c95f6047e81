// Query order: a spatially coherent ordering of the manifold points of one
// (library variable, E, tau), so that the query tiles of the fused kernel --
// consecutive runs of this order -- hold nearby points.  Nearby queries pass
// the running top-(E+1) thresholds on many of the same library points, so a
// warp takes the rare insertion path far less often than with queries in time
// order.  The order changes which tile a query belongs to and nothing else:
// every query's neighbours and prediction are the same in any order.
//
// Key: Morton interleave of all E coordinates, each quantised to floor(30/E) bits
// over the series' [min, max]; ties (and the key's low half) by the manifold
// index m, so the order is a deterministic function of the series.  With the
// first three coordinates only, neighbours in the order could lie apart in the
// others: rows of E = 10 tables (N = 10^4) then compare 234 of 313 chunks
// instead of 117, and a warp's brute-force queries at E = 6 meet 49 of 150
// library points instead of 12.
// One CTA per (variable, E, tau) sorts in shared memory when N_m <=
// kOrderMaxSort (a radix sort of the codes, a bitonic network for the shortest);
// a longer manifold is sorted by one CTA too: runs of kOrderMaxSort points, then
// merged pairwise in global scratch (merge path: every thread finds its output
// range by a binary search on the diagonal), which gives the same order.
#include <float.h>
#include <stdint.h>

#include "ccm_internal.h"
#include "launch.cuh"

namespace ccm {
namespace {

constexpr int kOrderThreads = 1024;

__device__ __forceinline__ uint32_t quantise(float c, float lo, float inv, int bits) {
  const float u = (c - lo) * inv;  // in [0, 1] up to rounding
  const float v = fmaxf(floorf(u * (float)(1u << bits)), 0.f);
  return min((uint32_t)v, (1u << bits) - 1u);  // as integers: 2^30 - 1 is no float
}

// Series range of job jb (block-wide min/max).
__device__ void series_range(const float* s, int64_t n, float* lo_out, float* hi_out) {
  __shared__ float s_lo[32], s_hi[32];
  float lo = FLT_MAX, hi = -FLT_MAX;
  for (int64_t t = threadIdx.x; t < n; t += blockDim.x) {
    lo = fminf(lo, s[t]);
    hi = fmaxf(hi, s[t]);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if ((threadIdx.x & 31) == 0) {
    s_lo[threadIdx.x >> 5] = lo;
    s_hi[threadIdx.x >> 5] = hi;
  }
  __syncthreads();
  lo = s_lo[0];
  hi = s_hi[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
    lo = fminf(lo, s_lo[w]);
    hi = fmaxf(hi, s_hi[w]);
  }
  __syncthreads();
  *lo_out = lo;
  *hi_out = hi;
}

// Sort key of manifold point q: (Morton code << 32) | q.  The code interleaves
// the top 30/E bits of every coordinate, the newest first.
__device__ __forceinline__ unsigned long long morton_key(const float* s, int off, int tau, int E,
                                                         float lo, float inv, int q) {
  const int t = q + off, bits = 30 / E;
  uint32_t code = 0u;
  for (int e = 0; e < E; ++e) {
    const uint32_t c = quantise(s[t - e * tau], lo, inv, bits);
    for (int b = 0; b < bits; ++b) code |= ((c >> b) & 1u) << (b * E + E - 1 - e);
  }
  return ((unsigned long long)code << 32) | (unsigned)q;
}

// Shared memory of radix_sort for up to n keys: codes, two index arrays, the
// warps' digit counts.
constexpr int kDigits = 256;
constexpr int kOrderWarps = kOrderThreads / 32;
size_t radix_smem(int n) {
  return (size_t)n * (4 + 2 + 2) + (size_t)kDigits * kOrderWarps * 4 + 64;
}
constexpr int kBitonicMax = 512;  // shorter manifolds: a bitonic network has fewer barriers

struct RadixBuffers {
  uint32_t* code;   // [n]
  uint16_t *a, *b;  // [n] each
  uint32_t* count;  // [warp][digit]
};
__device__ __forceinline__ RadixBuffers radix_buffers(unsigned char* smem, int n) {
  RadixBuffers r;
  r.count = reinterpret_cast<uint32_t*>(smem);
  r.code = r.count + kDigits * kOrderWarps;
  r.a = reinterpret_cast<uint16_t*>(r.code + n);
  r.b = r.a + n;
  return r;
}

// Sorts the indices 0 .. n-1 by code (30 bits), ties by index, by the whole
// block: four stable passes over eight-bit digits.  A warp owns a contiguous
// run of the sequence and takes it 32 at a time: lanes with the same digit find
// each other (match), so the digit's count advances once and the lanes' order
// is kept.  Returns the sorted index array.  16384 codes took 185 us as a
// bitonic network of 105 steps with a barrier each; 10000 take 58 us here with the
// codes and the range.
__device__ const uint16_t* radix_sort(const RadixBuffers& r, int n) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ uint32_t s_sum[kOrderWarps];
  const int seg = ((n + kOrderWarps - 1) / kOrderWarps + 31) / 32 * 32;
  const int q0 = min(n, warp * seg), q1 = min(n, q0 + seg);
  uint16_t *src = r.a, *dst = r.b;
  for (int q = tid; q < n; q += kOrderThreads) src[q] = (uint16_t)q;
  uint32_t* mine = r.count + warp * kDigits;
  for (int shift = 0; shift < 30; shift += 8) {
    for (int i = tid; i < kDigits * kOrderWarps; i += kOrderThreads) r.count[i] = 0u;
    __syncthreads();
    for (int q = q0 + lane; q - lane < q1; q += 32) {
      const bool in = q < q1;
      const uint32_t d = in ? (r.code[src[q]] >> shift) & (kDigits - 1) : kDigits;
      const unsigned same = __match_any_sync(0xffffffffu, d);
      if (in && lane == __ffs(same) - 1) mine[d] += (uint32_t)__popc(same);
      __syncwarp();
    }
    __syncthreads();
    // exclusive scan over (digit, warp): thread t takes eight warps of a digit
    const int d = tid >> 2, w0 = (tid & 3) * 8;
    uint32_t v[8], sum = 0u;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      v[i] = r.count[(w0 + i) * kDigits + d];
      sum += v[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    uint32_t before = s_sum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, before, o);
      if (lane >= o) before += y;
    }
    before = __shfl_sync(0xffffffffu, before, warp) - s_sum[warp];
    before += incl - sum;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      r.count[(w0 + i) * kDigits + d] = before;
      before += v[i];
    }
    __syncthreads();
    for (int q = q0 + lane; q - lane < q1; q += 32) {
      const bool in = q < q1;
      const uint16_t id = in ? src[q] : (uint16_t)0;
      const uint32_t dg = in ? (r.code[id] >> shift) & (kDigits - 1) : kDigits;
      const unsigned same = __match_any_sync(0xffffffffu, dg);
      const uint32_t at = in ? mine[dg] : 0u;
      __syncwarp();
      if (in) {
        dst[at + __popc(same & ((1u << lane) - 1u))] = id;
        if (lane == __ffs(same) - 1) mine[dg] = at + (uint32_t)__popc(same);
      }
      __syncwarp();
    }
    __syncthreads();
    uint16_t* t = src;
    src = dst;
    dst = t;
  }
  return src;
}

// Ascending bitonic sort of n2 (a power of two) keys in shared memory.
__device__ void bitonic_sort(unsigned long long* k, int n2) {
  for (int size = 2; size <= n2; size <<= 1) {
    for (int jj = size >> 1; jj > 0; jj >>= 1) {
      for (int q = threadIdx.x; q < n2; q += blockDim.x) {
        const int p = q ^ jj;
        if (p > q) {
          const unsigned long long a = k[q], b = k[p];
          const bool up = (q & size) == 0;
          if ((a > b) == up) {
            k[q] = b;
            k[p] = a;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Preparation of one target series (SeriesJob), by one CTA: the power of two
// 2^(kScaleBits - e), e the exponent of the series' largest magnitude (clamped so
// that it is a normal number; 1 for an all-zero or non-finite series), and its
// column of the time-major copy.
__device__ void prepare_series(const float* series, const SeriesJob& jb, SeriesScale* scales, float* st) {
  const float* s = series + jb.off;
  float lo, hi;
  series_range(s, jb.n, &lo, &hi);
  const float top = fmaxf(fabsf(lo), fabsf(hi));
  const float deep = __fmul_rn(top, __uint_as_float((uint32_t)(127 - kDeepBits) << 23));
  bool small = false;
  for (int64_t t = threadIdx.x; t < jb.n; t += blockDim.x) small |= s[t] != 0.f && fabsf(s[t]) < deep;
  small = __syncthreads_or(small);
  if (threadIdx.x == 0) {
    const int e = (int)((__float_as_uint(top) >> 23) & 0xffu) - 127;  // -127: zero or subnormal
    scales[jb.scale].scale = (top == 0.f || e == 128)
                                 ? 1.f
                                 : __uint_as_float((uint32_t)(127 + min(kScaleBits - e, 127)) << 23);
    scales[jb.scale].least_b2 = small ? 0.f : __uint_as_float(1u);
  }
  if (jb.st_off >= 0)
    for (int64_t t = threadIdx.x; t < jb.n; t += blockDim.x) st[jb.st_off + t * jb.st_stride] = s[t];
}

__global__ void __launch_bounds__(kOrderThreads)
order_kernel(const float* series, const OrderJob* jobs, int64_t n_jobs, int32_t* order,
             int32_t* inverse, unsigned long long* scratch, const SeriesJob* series_jobs, SeriesScale* scales, float* st) {
  extern __shared__ __align__(16) unsigned char s_order[];
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(s_order);
  chain_begin();
  if (blockIdx.x >= n_jobs) {
    prepare_series(series, series_jobs[blockIdx.x - n_jobs], scales, st);
    return;
  }
  const OrderJob jb = jobs[blockIdx.x];
  const float* s = series + jb.series_off + (int64_t)jb.j * jb.n;
  const int n_m = jb.n_m, E = jb.E, tau = jb.tau, off = (E - 1) * tau;
  // position q of the query order holds manifold point m
  auto put = [&](int q, int m) {
    order[jb.order_off + q] = m;
    if (inverse) inverse[jb.order_off + m] = q;
  };
  if (n_m > kOrderMaxSort && jb.scratch_off < 0) {  // no scratch: time order
    for (int m = threadIdx.x; m < n_m; m += blockDim.x) put(m, m);
    return;
  }
  float lo, hi;
  series_range(s, jb.n, &lo, &hi);
  const float inv = (hi > lo) ? 1.f / (hi - lo) : 0.f;
  if (n_m > kBitonicMax && n_m <= kOrderMaxSort) {
    const RadixBuffers r = radix_buffers(s_order, n_m);
    for (int q = threadIdx.x; q < n_m; q += blockDim.x)
      r.code[q] = (uint32_t)(morton_key(s, off, tau, E, lo, inv, q) >> 32);
    const uint16_t* sorted = radix_sort(r, n_m);
    for (int q = threadIdx.x; q < n_m; q += blockDim.x) put(q, sorted[q]);
    return;
  }
  if (n_m <= kOrderMaxSort) {
    int n2 = 1;
    while (n2 < n_m) n2 <<= 1;
    for (int q = threadIdx.x; q < n2; q += blockDim.x)
      s_key[q] = (q < n_m) ? morton_key(s, off, tau, E, lo, inv, q) : ~0ull;
    __syncthreads();
    bitonic_sort(s_key, n2);
    for (int q = threadIdx.x; q < n_m; q += blockDim.x) put(q, (int32_t)(s_key[q] & 0xffffffffu));
    return;
  }
  // Long manifold: sorted runs of kOrderMaxSort keys, then pairwise merges.
  unsigned long long* buf[2] = {scratch + jb.scratch_off, scratch + jb.scratch_off + n_m};
  for (int r0 = 0; r0 < n_m; r0 += kOrderMaxSort) {
    const int len = min(kOrderMaxSort, n_m - r0);
    const RadixBuffers r = radix_buffers(s_order, len);
    for (int q = threadIdx.x; q < len; q += blockDim.x)
      r.code[q] = (uint32_t)(morton_key(s, off, tau, E, lo, inv, r0 + q) >> 32);
    const uint16_t* sorted = radix_sort(r, len);
    for (int q = threadIdx.x; q < len; q += blockDim.x)
      buf[0][r0 + q] = ((unsigned long long)r.code[sorted[q]] << 32) | (unsigned)(r0 + sorted[q]);
    __syncthreads();
  }
  int src = 0;
  for (int width = kOrderMaxSort; width < n_m; width <<= 1, src ^= 1) {
    const unsigned long long* in = buf[src];
    unsigned long long* dst = buf[src ^ 1];
    for (int b0 = 0; b0 < n_m; b0 += 2 * width) {
      const int a_len = min(width, n_m - b0);
      const int b_len = max(0, min(width, n_m - b0 - width));
      const unsigned long long* A = in + b0;
      const unsigned long long* B = in + b0 + a_len;
      const int total = a_len + b_len;
      const int per = (total + blockDim.x - 1) / blockDim.x;
      const int k0 = min(total, (int)threadIdx.x * per), k1 = min(total, k0 + per);
      if (k0 < k1) {
        // merge path: i keys from A and k0 - i from B precede output k0 (keys are distinct)
        int lo_i = max(0, k0 - b_len), hi_i = min(k0, a_len);
        while (lo_i < hi_i) {
          const int mid = (lo_i + hi_i) >> 1;
          if (A[mid] < B[k0 - 1 - mid]) lo_i = mid + 1;
          else hi_i = mid;
        }
        int i = lo_i, jv = k0 - lo_i;
        for (int k = k0; k < k1; ++k) {
          const bool take_a = jv >= b_len || (i < a_len && A[i] < B[jv]);
          dst[b0 + k] = take_a ? A[i++] : B[jv++];
        }
      }
    }
    __syncthreads();
  }
  for (int q = threadIdx.x; q < n_m; q += blockDim.x) put(q, (int32_t)(buf[src][q] & 0xffffffffu));
}

}  // namespace

cudaError_t order_prepare() {
  return cudaFuncSetAttribute(order_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)radix_smem(kOrderMaxSort));
}

cudaError_t launch_order(const float* series, const OrderJob* jobs, int64_t n_jobs, int max_nm,
                         int32_t* order, int32_t* inverse, unsigned long long* scratch,
                         const SeriesJob* series_jobs, int64_t n_series_jobs, SeriesScale* scales,
                         float* st, LaunchStream s) {
  if (n_jobs + n_series_jobs <= 0) return cudaSuccess;
  const size_t smem = max_nm <= kBitonicMax ? (size_t)kBitonicMax * sizeof(unsigned long long)
                                            : radix_smem(max_nm < kOrderMaxSort ? max_nm : kOrderMaxSort);
  return launch_chained(order_kernel, dim3((unsigned)(n_jobs + n_series_jobs)), kOrderThreads, smem, s,
                        series, jobs, n_jobs, order, inverse, scratch, series_jobs, scales, st);
}

}  // namespace ccm
