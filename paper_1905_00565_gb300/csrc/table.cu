// Distance indexing tables: the manifold's points in query order with their
// bounding boxes, and the dispatch of the build (table_build.cu) by E.
#include <math.h>
#include <stdint.h>

#include "ccm_internal.h"
#include "launch.cuh"

namespace ccm {
namespace {

constexpr int kPointThreads = 1024;  // one superchunk: 32 chunks of 32 points

// One CTA per superchunk: coordinates [chunk][E][32], the chunk boxes and the
// superchunk's box, and the smallest manifold index of each (TableJob).  A box's
// sides are (lo, hi) per coordinate,
// arrays over the boxes; NaN coordinates are left out of them, and positions
// past the manifold's end do not count.
__global__ void __launch_bounds__(kPointThreads)
table_points_kernel(const float* series, const TableJob* jobs, const int32_t* order,
                    float* points) {
  __shared__ float s_lo[32], s_hi[32];
  __shared__ int s_least[32];
  chain_begin();
  const TableJob jb = jobs[blockIdx.y];
  const int n_m = jb.n_m, E = jb.E, tau = jb.tau, off = (E - 1) * tau;
  const int n_chunks = (n_m + 31) >> 5, n_super = (n_chunks + 31) >> 5;
  const int super = blockIdx.x;
  if (super >= n_super) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int chunk = super * 32 + warp, pos = chunk * 32 + lane;
  const float* s = series + jb.series_off + (int64_t)jb.j * jb.n;
  const bool valid = pos < n_m;
  const int m = valid ? order[jb.order_off + pos] : 0;
  int32_t* least = reinterpret_cast<int32_t*>(points + jb.least_off);
  const int first = __reduce_min_sync(0xffffffffu, valid ? m : n_m);
  if (lane == 0) least[chunk] = s_least[warp] = first;
  __syncthreads();
  if (warp == 0) {
    const int all = __reduce_min_sync(0xffffffffu, s_least[lane]);
    if (lane == 0) least[n_super * 32 + super] = all;
  }
  for (int e = 0; e < E; ++e) {
    const float c = valid ? s[m + off - e * tau] : 0.f;
    if (chunk < n_chunks) points[jb.pts_off + ((int64_t)chunk * E + e) * 32 + lane] = c;
    const int n_sample = n_m / jb.sample, at = pos / jb.sample;
    if (pos == at * jb.sample + (jb.sample >> 1) && at < n_sample)
      points[jb.sample_off + (int64_t)e * n_sample + at] = c;
    float lo = valid ? c : INFINITY, hi = valid ? c : -INFINITY;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      points[jb.box_off + (int64_t)(2 * e) * n_super * 32 + chunk] = lo;
      points[jb.box_off + (int64_t)(2 * e + 1) * n_super * 32 + chunk] = hi;
      s_lo[warp] = lo;
      s_hi[warp] = hi;
    }
    __syncthreads();
    if (warp == 0) {
      lo = s_lo[lane];
      hi = s_hi[lane];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      }
      if (lane == 0) {
        points[jb.sbox_off + (int64_t)(2 * e) * n_super + super] = lo;
        points[jb.sbox_off + (int64_t)(2 * e + 1) * n_super + super] = hi;
      }
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_table_points(const float* series, const TableJob* jobs, int64_t n_jobs,
                                int max_nm, const int32_t* order, float* points, LaunchStream s) {
  for (int64_t at = 0; at < n_jobs; at += 65535) {
    const dim3 grid((unsigned)((max_nm + 1023) / 1024),
                    (unsigned)(n_jobs - at < 65535 ? n_jobs - at : 65535));
    const cudaError_t e =
        launch_chained(table_points_kernel, grid, kPointThreads, 0, s, series, jobs + at, order, points);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

#define CCM_FOR_E(X) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10)
#define CCM_CASE_PREPARE(EV) \
  if (const cudaError_t e = TableKernels<EV>::prepare(); e != cudaSuccess) return e;
#define CCM_CASE_LAUNCH(EV)                                                                     \
  case EV:                                                                                      \
    return TableKernels<EV>::launch(series, jobs, n_jobs, n_rows, max_nm, max_R, points, order, \
                                    inverse, table, table_dist, table_pairs, table_u16, err, s);

cudaError_t table_prepare() {
  CCM_FOR_E(CCM_CASE_PREPARE)
  return cudaSuccess;
}

cudaError_t launch_table_build(const float* series, const TableJob* jobs, int64_t n_jobs,
                               int64_t n_rows, int E, int max_nm, int max_R, const float* points,
                               const int32_t* order, const int32_t* inverse, void* table,
                               float* table_dist, int table_pairs, int table_u16, int32_t* err,
                               LaunchStream s) {
  if (n_jobs <= 0) return cudaSuccess;
  if (max_R > kTableMaxR) return cudaErrorInvalidValue;
  switch (E) { CCM_FOR_E(CCM_CASE_LAUNCH) }
  return cudaErrorInvalidValue;
}

}  // namespace ccm
