// Observed-value records, rho and the dispatch of the search kernels by E.
#include <float.h>

#include "ccm_internal.h"
#include "launch.cuh"
#include "moments.cuh"

namespace ccm {
namespace {

constexpr int kThreads = 256;
// CTAs of the FP64 kernels: one warp, so that few targets spread over the SMs (a
// warp's FP64 instruction takes 16 cycles of its SM's pipe).
constexpr int kSmallThreads = 32;
constexpr unsigned kFull = 0xffffffffu;

// Butterfly sum over the warp: every lane ends with the same bits (each
// level adds the same two values in either order).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(kFull, v, o));
  return v;
}

constexpr int kPer = kQT / 32;  // queries per lane

// Observed-value records (see ObsJob), one warp per tile: x_q is the target
// at the tile's manifold points (Sect. 2.1: the value the cross map
// predicts).  Two passes in FP64, then split into float pairs.
__global__ void __launch_bounds__(kSmallThreads) obs_kernel(const float* series, const int32_t* order,
                                                      const ObsJob* jobs, int64_t n_jobs,
                                                      int64_t n_tiles, const SeriesScale* scales,
                                                      float2* obs, ObsStat* obs_stat) {
  chain_begin();
  const int lane = threadIdx.x & 31;
  const int64_t n_warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < n_tiles;
       g += n_warps) {
    int64_t lo = 0, hi = n_jobs - 1;  // the job holding tile g: last obs_tile <= g
    while (lo < hi) {
      const int64_t mid = (lo + hi + 1) >> 1;
      if (jobs[mid].obs_tile <= g) lo = mid;
      else hi = mid - 1;
    }
    const ObsJob jb = jobs[lo];
    const int tile = (int)(g - jb.obs_tile);
    const int nq = min(kQT, jb.n_m - tile * kQT);
    const float* si = series + jb.series_off + (int64_t)jb.i * jb.n;
    const int32_t* ord = order + jb.order_off + (int64_t)tile * kQT;
    const int off = (jb.E - 1) * jb.tau;
    const SeriesScale sc = scales[jb.scale];
    const float scale = sc.scale;
    float s[kPer];
    double x[kPer];
    double sv = 0.0;
    bool inexact = false;  // the product of some value leaves FP32's normal range
#pragma unroll
    for (int c = 0; c < kPer; ++c) {
      const int q = lane + 32 * c;
      s[c] = (q < nq) ? si[ord[q] + off] : 0.f;
      const float scaled = __fmul_rn(s[c], scale);
      x[c] = (double)scaled;
      inexact |= s[c] != 0.f && fabsf(scaled) < FLT_MIN;
    }
    if (__builtin_expect(inexact, 0)) {
#pragma unroll
      for (int c = 0; c < kPer; ++c) x[c] = __dmul_rn((double)s[c], (double)scale);
    }
#pragma unroll
    for (int c = 0; c < kPer; ++c) sv = __dadd_rn(sv, x[c]);
    const double mx = __ddiv_rn(warp_sum(sv), (double)nq);
    double sxx = 0.0;
#pragma unroll
    for (int c = 0; c < kPer; ++c) {
      const int q = lane + 32 * c;
      const double a = (q < nq) ? __dsub_rn(x[c], mx) : 0.0;
      sxx = __fma_rn(a, a, sxx);
      const float h = __double2float_rn(a);
      const float2 v = make_float2(h, __double2float_rn(__dsub_rn(a, (double)h)));
      if (jb.a_step == 0) obs[jb.a_off + (int64_t)tile * kQT + obs_slot(q)] = v;
      else obs[jb.a_off + ((int64_t)tile * kQT + q) * jb.a_step] = v;
    }
    sxx = warp_sum(sxx);
    if (lane == 0) {
      ObsStat& o = obs_stat[g];
      o.mx = mx;
      o.sxx = sxx;
      o.series = sc;
    }
  }
}

// rho of one target: the tile moments merged.  With the grand means MX =
// sum(n_t mx_t)/N, the centred sums are exactly
//   Sxx = sum_t [Sxx_t + n_t (mx_t - MX)^2]   (likewise Syy, Sxy),
// a sum of non-negative terms (no cancellation).  kRhoLanes lanes (a whole warp
// for targets of more than kRhoNarrow tiles) take every so-many-th tile and are
// added in a fixed order, so rho does not depend on which CTA ran which tile, or
// when.  A launch of its own: FP64 instructions cost the same for one lane as
// for 32, and merging inside the search kernels kept whole warps on it (and a
// fence and a counter per tile).  Bound: the FP64 pipe for many targets, the
// loads' latency for few (four tiles' loads are in flight per lane).
constexpr int kRhoLanes = 4;
constexpr int kRhoNarrow = 96;
constexpr int kRhoAhead = 4;  // tiles a lane loads at once

template <int kLanes>
__device__ __forceinline__ double rho_sum(double v) {
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) v = __dadd_rn(v, __shfl_xor_sync(kFull, v, o));
  return v;
}

// A tile's mean of y and its centred sums, from its record (moments.cuh).
__device__ __forceinline__ double tile_mean(const float4& a, const float4& b, double n, double& b1,
                                            double& d) {
  if (b.w != 0.f) return word_pair(a.x, a.y);  // a record in FP64
  b1 = __dadd_rn((double)a.y, (double)a.z);  // sum(y - c)
  d = (n == (double)kQT) ? __dmul_rn(b1, 1.0 / kQT) : __ddiv_rn(b1, n);
  return __dadd_rn((double)a.x, d);
}
__device__ __forceinline__ void tile_moments(const float4& a, const float4& b, double n, double& my,
                                             double& syy, double& sxy) {
  double b1, d;
  my = tile_mean(a, b, n, b1, d);
  if (b.w != 0.f) {
    syy = word_pair(a.z, a.w);
    sxy = word_pair(b.x, b.y);
  } else {
    const double b2 = __dadd_rn((double)a.w, (double)b.x);
    syy = fmax(__fma_rn(-b1, d, b2), 0.0);
    sxy = __dadd_rn((double)b.y, (double)b.z);
  }
}

// rho of a target by kLanes lanes (lane `sub` of them); `active` false: the
// lanes only take part in the shuffles.  kKeep (at most kRhoAhead*kLanes tiles): the
// tiles' values are worked out once and stay in registers; else each of the two passes
// reads the records and works out what it needs.  10^5 targets of 16 tiles 154 -> 125
// us, of 4 tiles 76 -> 68, of 20 tiles (not kept) 180; a cell of N = 300, r = 400 62 ->
// 59.5 us (its rho is a chain of instructions that the SMs meet for the first time).
template <int kLanes, bool kKeep>
__device__ __forceinline__ double target_rho(int n_tiles, int n_m, const float4* base,
                                             const ObsStat* stat, int sub, bool active) {
  constexpr int kAhead = kRhoAhead;
  struct Tile {
    float4 a, b;
    double mx, sxx;
  };
  struct Kept {
    double n, my, syy, sxy;
  };
  auto load = [&](int q0, Tile (&t)[kAhead]) {
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int q = q0 + i * kLanes;
      if (q < n_tiles) {
        t[i].a = base[2 * q];
        t[i].b = base[2 * q + 1];
        t[i].mx = __ldg(&stat[q].mx);
        t[i].sxx = __ldg(&stat[q].sxx);
      }
    }
  };
  auto count = [&](int q) { return (double)min(kQT, n_m - q * kQT); };
  Tile t[kAhead];
  Kept kept[kAhead];
  double SX = 0.0, SY = 0.0, b1, d;
  for (int q0 = sub; active && q0 < n_tiles; q0 += kAhead * kLanes) {
    load(q0, t);
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int q = q0 + i * kLanes;
      if (q >= n_tiles) break;
      const double n = count(q);
      SX = __fma_rn(n, t[i].mx, SX);
      if (kKeep) {
        kept[i].n = n;
        tile_moments(t[i].a, t[i].b, n, kept[i].my, kept[i].syy, kept[i].sxy);
        SY = __fma_rn(n, kept[i].my, SY);
      } else {
        SY = __fma_rn(n, tile_mean(t[i].a, t[i].b, n, b1, d), SY);
      }
    }
    if (kKeep) break;
  }
  const double inv = (double)n_m;
  const double MX = __ddiv_rn(rho_sum<kLanes>(SX), inv), MY = __ddiv_rn(rho_sum<kLanes>(SY), inv);
  double SXX = 0.0, SYY = 0.0, SXY = 0.0;
  for (int q0 = sub; active && q0 < n_tiles; q0 += kAhead * kLanes) {
    if (!kKeep) load(q0, t);
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int q = q0 + i * kLanes;
      if (q >= n_tiles) break;
      Kept k = kept[i];
      if (!kKeep) {
        k.n = count(q);
        tile_moments(t[i].a, t[i].b, k.n, k.my, k.syy, k.sxy);
      }
      const double dy = __dsub_rn(k.my, MY), dx = __dsub_rn(t[i].mx, MX);
      const double wx = __dmul_rn(k.n, dx);
      SXX = __fma_rn(wx, dx, __dadd_rn(SXX, t[i].sxx));
      SYY = __fma_rn(__dmul_rn(k.n, dy), dy, __dadd_rn(SYY, k.syy));
      SXY = __fma_rn(wx, dy, __dadd_rn(SXY, k.sxy));
    }
    if (kKeep) break;
  }
  SXX = rho_sum<kLanes>(SXX);
  SYY = rho_sum<kLanes>(SYY);
  SXY = rho_sum<kLanes>(SXY);
  return (SXX > 0.0 && SYY > 0.0) ? __ddiv_rn(SXY, __dsqrt_rn(__dmul_rn(SXX, SYY))) : nan("");
}

// rho of a target of at most kRhoNarrow tiles by a whole warp, to the same bits as by
// kRhoLanes lanes: the tiles' values by 32 lanes at once, then every lane adds up
// those of its narrow lane (lane mod kRhoLanes) in that lane's order.
struct TileRow {
  double n, mx, my, sxx, syy, sxy, wx, dx, wy, dy;
};
__device__ __forceinline__ double wide_rho(int n_tiles, int n_m, const float4* base,
                                           const ObsStat* stat, TileRow* rows) {
  const int lane = threadIdx.x & 31, sub = lane & (kRhoLanes - 1);
  for (int q = lane; q < n_tiles; q += 32) {
    TileRow& t = rows[q];
    const float4 a = base[2 * q], b = base[2 * q + 1];
    t.n = (double)min(kQT, n_m - q * kQT);
    t.mx = stat[q].mx;
    t.sxx = stat[q].sxx;
    tile_moments(a, b, t.n, t.my, t.syy, t.sxy);
  }
  __syncwarp();
  double SX = 0.0, SY = 0.0;
#pragma unroll 4
  for (int q = sub; q < n_tiles; q += kRhoLanes) {
    SX = __fma_rn(rows[q].n, rows[q].mx, SX);
    SY = __fma_rn(rows[q].n, rows[q].my, SY);
  }
  const double inv = (double)n_m;
  const double MX = __ddiv_rn(rho_sum<kRhoLanes>(SX), inv), MY = __ddiv_rn(rho_sum<kRhoLanes>(SY), inv);
  for (int q = lane; q < n_tiles; q += 32) {
    TileRow& t = rows[q];
    t.dx = __dsub_rn(t.mx, MX);
    t.dy = __dsub_rn(t.my, MY);
    t.wx = __dmul_rn(t.n, t.dx);
    t.wy = __dmul_rn(t.n, t.dy);
  }
  __syncwarp();
  double SXX = 0.0, SYY = 0.0, SXY = 0.0;
#pragma unroll 4
  for (int q = sub; q < n_tiles; q += kRhoLanes) {
    const TileRow& t = rows[q];
    SXX = __fma_rn(t.wx, t.dx, __dadd_rn(SXX, t.sxx));
    SYY = __fma_rn(t.wy, t.dy, __dadd_rn(SYY, t.syy));
    SXY = __fma_rn(t.wx, t.dy, __dadd_rn(SXY, t.sxy));
  }
  SXX = rho_sum<kRhoLanes>(SXX);
  SYY = rho_sum<kRhoLanes>(SYY);
  SXY = rho_sum<kRhoLanes>(SXY);
  return (SXX > 0.0 && SYY > 0.0) ? __ddiv_rn(SXY, __dsqrt_rn(__dmul_rn(SXX, SYY))) : nan("");
}

// Few targets of more tiles than a narrow lane takes at once: a warp each.  A narrow
// lane of N = 20000 walks 20 tiles twice, four at a time: 100 targets 32 us on 13
// SMs, 16.5 us here.  From kRhoFew targets on the pipe time of whole warps' FP64
// instructions counts more; with 16 tiles or less the narrow lanes are as quick and a
// launch of fewer CTAs is shorter (N = 1000, 400 targets: a cell 80.5 against 82.1 us).
constexpr int64_t kRhoFew = 1024;
__global__ void __launch_bounds__(kSmallThreads) rho_few_kernel(const UnitDesc* units,
                                                                const TargetDesc* targets,
                                                                const float4* partials,
                                                                const ObsStat* obs_stat, double* rho) {
  __shared__ TileRow rows[kRhoNarrow];
  chain_begin();
  const TargetDesc tg = targets[blockIdx.x];
  const UnitDesc& u = units[tg.unit];
  const float4* base = partials + 2 * (u.part_off + (blockIdx.x - u.tgt_off) * u.n_tiles);
  const ObsStat* stat = obs_stat + tg.obs_tile;
  const double r = u.n_tiles <= kRhoNarrow
                       ? wide_rho(u.n_tiles, u.n_m, base, stat, rows)
                       : target_rho<32, false>(u.n_tiles, u.n_m, base, stat, threadIdx.x & 31, true);
  if (threadIdx.x == 0) rho[tg.out_idx] = r;
}

__global__ void __launch_bounds__(kSmallThreads) rho_kernel(const UnitDesc* units,
                                                      const TargetDesc* targets,
                                                      int64_t n_targets, const float4* partials,
                                                      const ObsStat* obs_stat, double* rho) {
  chain_begin();
  const int lane = threadIdx.x & 31, sub = lane & (kRhoLanes - 1);
  const int64_t first = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x - lane) / kRhoLanes;
  const int64_t g = first + lane / kRhoLanes;  // this lane's target
  const int64_t at = g < n_targets ? g : n_targets - 1;  // whole warps shuffle
  auto of = [&](int64_t i, TargetDesc& tg, int& n_tiles, int& n_m) {
    tg = targets[i];
    const UnitDesc& u = units[tg.unit];
    n_tiles = u.n_tiles;
    n_m = u.n_m;
    return partials + 2 * (u.part_off + (i - u.tgt_off) * n_tiles);
  };
  TargetDesc tg;
  int n_tiles, n_m;
  const float4* base = of(at, tg, n_tiles, n_m);
  const bool narrow = n_tiles <= kRhoNarrow;
  if (__any_sync(kFull, narrow)) {
    const double r =
        __all_sync(kFull, n_tiles <= kRhoAhead * kRhoLanes)
            ? target_rho<kRhoLanes, true>(n_tiles, n_m, base, obs_stat + tg.obs_tile, sub, true)
            : target_rho<kRhoLanes, false>(n_tiles, n_m, base, obs_stat + tg.obs_tile, sub, narrow);
    if (narrow && sub == 0 && g < n_targets) rho[tg.out_idx] = r;
  }
  if (__all_sync(kFull, narrow)) return;
  for (int i = 0; i < 32 / kRhoLanes && first + i < n_targets; ++i) {
    base = of(first + i, tg, n_tiles, n_m);
    if (n_tiles <= kRhoNarrow) continue;  // the same for the whole warp
    const double r = target_rho<32, false>(n_tiles, n_m, base, obs_stat + tg.obs_tile, lane, true);
    if (lane == 0) rho[tg.out_idx] = r;
  }
}

}  // namespace

int knn_block_threads() { return kThreads; }
int knn_queries_per_thread() { return 1; }

#define CCM_FOR_E(X) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10)
#define CCM_CASE_PREPARE(EV)                                             \
  if (const cudaError_t e = KnnKernels<EV>::prepare(); e != cudaSuccess) return e;
#define CCM_CASE_PREPARE_TABLE(EV)                                       \
  if (const cudaError_t e = KnnKernels<EV>::prepare_table(); e != cudaSuccess) return e;
#define CCM_CASE_PREPARE_SCAN(EV)                                        \
  if (const cudaError_t e = KnnKernels<EV>::prepare_scan(); e != cudaSuccess) return e;
#define CCM_CASE_PREPARE_GROUP(EV)                                       \
  if (const cudaError_t e = KnnKernels<EV>::prepare_group(); e != cudaSuccess) return e;
#define CCM_CASE_LAUNCH_GROUP(EV) \
  case EV: return KnnKernels<EV>::launch_group(p, max_nm, grid, s);
#define CCM_CASE_LAUNCH_SCAN(EV) \
  case EV: return KnnKernels<EV>::launch_scan(p, max_nm, grid, s);
#define CCM_CASE_OCCUPANCY(EV) \
  case EV: return KnnKernels<EV>::occupancy(ctas);
#define CCM_CASE_LAUNCH(EV) \
  case EV: return KnnKernels<EV>::launch(p, lanes, grid, s);
#define CCM_CASE_LAUNCH_TABLE(EV) \
  case EV: return KnnKernels<EV>::launch_table(p, max_nm, lanes, grid, s);

cudaError_t knn_prepare() {
  CCM_FOR_E(CCM_CASE_PREPARE)
  return cudaSuccess;
}
cudaError_t knn_table_prepare() {
  CCM_FOR_E(CCM_CASE_PREPARE_TABLE)
  return cudaSuccess;
}
cudaError_t knn_scan_prepare() {
  CCM_FOR_E(CCM_CASE_PREPARE_SCAN)
  return cudaSuccess;
}
cudaError_t launch_knn_scan(const KnnParams& p, int E, int max_nm, int grid, LaunchStream s) {
  switch (E) { CCM_FOR_E(CCM_CASE_LAUNCH_SCAN) }
  return cudaErrorInvalidValue;
}
cudaError_t knn_group_prepare() {
  CCM_FOR_E(CCM_CASE_PREPARE_GROUP)
  return cudaSuccess;
}
cudaError_t launch_knn_group(const KnnParams& p, int E, int max_nm, int grid, LaunchStream s) {
  switch (E) { CCM_FOR_E(CCM_CASE_LAUNCH_GROUP) }
  return cudaErrorInvalidValue;
}
cudaError_t knn_occupancy(int E, int* ctas) {
  switch (E) { CCM_FOR_E(CCM_CASE_OCCUPANCY) }
  return cudaErrorInvalidValue;
}
cudaError_t launch_knn(const KnnParams& p, int E, bool lanes, int grid, LaunchStream s) {
  switch (E) { CCM_FOR_E(CCM_CASE_LAUNCH) }
  return cudaErrorInvalidValue;
}
cudaError_t knn_table_occupancy(int max_nm, bool lanes, int* ctas) {
  return KnnKernels<kMaxE>::occupancy_table(max_nm, lanes, ctas);
}
cudaError_t launch_knn_table(const KnnParams& p, int E, int max_nm, bool lanes, int grid,
                             LaunchStream s) {
  switch (E) { CCM_FOR_E(CCM_CASE_LAUNCH_TABLE) }
  return cudaErrorInvalidValue;
}

cudaError_t launch_obs(const float* series, const int32_t* order, const ObsJob* jobs,
                       int64_t n_jobs, int64_t n_tiles, const SeriesScale* scales, float2* obs,
                       ObsStat* obs_stat, LaunchStream s) {
  if (n_jobs <= 0 || n_tiles <= 0) return cudaSuccess;
  const int64_t want = (n_tiles + kSmallThreads / 32 - 1) / (kSmallThreads / 32);  // a warp per tile
  const int64_t blocks = want < (1 << 20) ? want : 1 << 20;
  return launch_chained(obs_kernel, dim3((unsigned)blocks), kSmallThreads, 0, s, series, order, jobs,
                        n_jobs, n_tiles, scales, obs, obs_stat);
}

cudaError_t launch_rho(const UnitDesc* units, const TargetDesc* targets, int64_t n_targets,
                       int max_tiles, const float4* partials, const ObsStat* obs_stat, double* rho,
                       LaunchStream s) {
  if (n_targets <= 0) return cudaSuccess;
  if (n_targets <= kRhoFew && max_tiles > kRhoAhead * kRhoLanes)
    return launch_chained(rho_few_kernel, dim3((unsigned)n_targets), kSmallThreads, 0, s, units, targets,
                          partials, obs_stat, rho);
  const int64_t blocks = (n_targets * kRhoLanes + kSmallThreads - 1) / kSmallThreads;
  return launch_chained(rho_kernel, dim3((unsigned)blocks), kSmallThreads, 0, s, units, targets,
                        n_targets, partials, obs_stat, rho);
}

}  // namespace ccm
