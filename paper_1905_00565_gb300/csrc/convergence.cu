// Convergence decision on the rho grid (paper Sect. 1: cross-map skill should
// rise with the library size L, judged over the r realizations; the paper
// states no test, the one used here is a one-sided Jonckheere-Terpstra trend
// test over the L groups).
//
// One CTA per (pair, E, tau) row of rho [rows][n_L][r]: the row is staged in
// shared memory with the L groups in increasing L and every group is sorted;
// then each finite member y adds, for every earlier group, twice the number of
// its members below y and once those equal to y (a binary search), so 2J is an
// exact integer.  Non-finite rho (a realization with zero variance) are
// left out.  Thread 0 forms E[J], Var[J] (no tie correction), z and the group
// means (summed in realization order) with explicit
// round-to-nearest operations in a fixed order: group sizes summed in
// increasing L, then E[J], Var[J] and z, so the result depends on nothing but
// the row.
#include <math.h>
#include <stdint.h>

#include "ccm_internal.h"

namespace ccm {
namespace {

constexpr int kConvThreads = 256;

using u64 = unsigned long long;

// A finite double as an integer that orders the same way (negative values
// complemented, the sign bit set on the others; -0 counts as +0).  GB300's
// FP64 pipe takes two lanes per SM per clock and a comparison goes through it,
// so sorting and searching doubles is bound by it; the integers run on the ALU.
constexpr u64 kMissing = ~0ull;  // a non-finite realization: above every finite key
__device__ __forceinline__ u64 order_key(u64 bits) {
  if (((bits >> 52) & 0x7ffull) == 0x7ffull) return kMissing;
  if (bits == 0x8000000000000000ull) bits = 0ull;
  return (bits >> 63) ? ~bits : bits | 0x8000000000000000ull;
}

// Ascending sort, by the whole block, of each of n_g groups of n keys
// (group g at v + g*n): a bitonic network whose comparators all put the
// smaller key at the lower index (the first step of every merge compares
// mirrored positions), over the next power of two 2^lg with virtual largest
// keys beyond n, so positions at or above n never take part.  One barrier per
// step.
__device__ void block_sort_groups(u64* v, int n_g, int n, int lg) {
  const int lh = lg - 1, pairs = (lg > 0) ? n_g << lh : 0;
  for (int lk = 1; lk <= lg; ++lk) {
    for (int lj = lk - 1; lj >= 0; --lj) {
      const int jj = 1 << lj;
      const int mirror = (lj == lk - 1) ? 2 * jj - 1 : 0;
      for (int t = threadIdx.x; t < pairs; t += blockDim.x) {
        // pair of this step: block of size 2*jj, offset inside the half
        const int g = t >> lh, tp = t & ((1 << lh) - 1);
        const int off = tp & (jj - 1), lo = ((tp >> lj) << (lj + 1)) + off;
        const int j = mirror ? lo - 2 * off + mirror : lo + jj;
        if (j < n) {
          u64* w = v + g * n;
          const u64 a = w[lo], c = w[j];
          if (c < a) {
            w[lo] = c;
            w[j] = a;
          }
        }
      }
      __syncthreads();
    }
  }
}

__device__ __forceinline__ void order_pair(u64& a, u64& b) {
  const u64 lo = a < b ? a : b;
  b = a < b ? b : a;
  a = lo;
}

// The same network over 32*P keys in one warp's registers, key e = lane*P + i:
// steps shorter than P stay in a lane, the others exchange with another lane
// (the mirrored first step of a merge also mirrors the lane's registers).
template <int P>
__device__ __forceinline__ void warp_sort(u64 (&k)[P]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int size = 2; size <= 32 * P; size <<= 1) {
#pragma unroll
    for (int jj = size / 2; jj > 0; jj >>= 1) {
      const bool mirror = jj == size / 2;
      if (jj >= P) {
        const int x = mirror ? 2 * (jj / P) - 1 : jj / P;
        const bool low = (lane & (jj / P)) == 0;
        u64 other[P];
#pragma unroll
        for (int i = 0; i < P; ++i)
          other[i] = __shfl_xor_sync(0xffffffffu, k[mirror ? P - 1 - i : i], x);
#pragma unroll
        for (int i = 0; i < P; ++i) k[i] = ((other[i] < k[i]) == low) ? other[i] : k[i];
      } else {
#pragma unroll
        for (int i = 0; i < P; ++i) {
          const int j = mirror ? i + 2 * jj - 1 - 2 * (i & (jj - 1)) : i + jj;
          if ((i & jj) == 0) order_pair(k[i], k[j]);
        }
      }
    }
  }
}

// Reads the groups into shared memory as sorted keys, one warp per group (r <=
// 32*P): no barrier, and a third of the instructions of the block-wide network.
template <int P>
__device__ __forceinline__ void load_sorted(const u64* bits, const ConvOrder& ord, int n_L, int r,
                                            u64* s_key, int* s_cnt) {
  const int lane = threadIdx.x & 31;
  for (int g = threadIdx.x >> 5; g < n_L; g += kConvThreads / 32) {
    const u64* src = bits + (int64_t)ord.group[g] * r;
    u64 k[P];
    int missing = 0;
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const int e = lane + 32 * i;
      k[i] = e < r ? order_key(src[e]) : kMissing;
      missing += (e < r && k[i] == kMissing) ? 1 : 0;
    }
    missing = __reduce_add_sync(0xffffffffu, missing);
    if (lane == 0) s_cnt[g] = r - missing;
    warp_sort<P>(k);
#pragma unroll
    for (int i = 0; i < P; ++i)
      if (lane * P + i < r) s_key[g * r + lane * P + i] = k[i];
  }
}

// Bound: issue (the searches, then the sorts).  12096 rows of 8 groups of 250
// take 0.73 ms; with double comparisons (FP64 pipe), two searches per (member,
// earlier group) and the means summed in front of a barrier they took 4.03 ms,
// with integer keys but the block-wide sort for every r 1.21 ms.
__global__ void __launch_bounds__(kConvThreads)
convergence_kernel(const double* rho, int32_t n_L, int32_t r, ConvOrder ord, double z_crit,
                   ConvergenceRow* out) {
  extern __shared__ u64 s_key[];              // [n_L][r], groups in increasing L
  __shared__ u64 s_j2[kConvThreads / 32];
  __shared__ int s_cnt[kMaxConvGroups];
  const int tid = threadIdx.x;
  const int64_t row = blockIdx.x;
  const int T = n_L * r;
  const double* src = rho + row * (int64_t)T;
  const u64* bits = reinterpret_cast<const u64*>(src);
  if (r <= 64) {
    load_sorted<2>(bits, ord, n_L, r, s_key, s_cnt);
  } else if (r <= 256) {
    load_sorted<8>(bits, ord, n_L, r, s_key, s_cnt);
  } else {  // longer groups (few rows have them): sorted in place by the whole block
    for (int g = tid; g < n_L; g += kConvThreads) s_cnt[g] = r;
    __syncthreads();
    for (int i = tid; i < T; i += kConvThreads) {
      const int g = i / r, k = i - g * r;
      const u64 x = order_key(bits[(int64_t)ord.group[g] * r + k]);
      s_key[i] = x;
      if (x == kMissing) atomicSub(&s_cnt[g], 1);  // sorts last and is not counted
    }
    __syncthreads();
    int lg = 0;
    while ((1 << lg) < r) ++lg;
    block_sort_groups(s_key, n_L, r, lg);
  }
  __syncthreads();
  int top = 1;  // the largest power of two within r
  while (2 * top <= r) top <<= 1;
  // 2J: for each finite y, the members of earlier groups below it (2 each) and
  // equal to it (1 each): one branch-free binary search per earlier group, four
  // groups at a time so that their loads overlap, and a second one for the
  // (rare) equal keys.
  u64 j2 = 0ull;
  for (int i = tid; i < T; i += kConvThreads) {
    const int g = i / r;
    if (i - g * r >= s_cnt[g]) continue;  // a non-finite realization
    const u64 y = s_key[i];
    for (int h0 = 0; h0 < g; h0 += 4) {
      int pos[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) pos[u] = 0;
      for (int step = top; step > 0; step >>= 1) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = pos[u] + step;  // missing keys lie above y: no need for the count
          if (h0 + u < g && p <= r && s_key[(h0 + u) * r + p - 1] < y) pos[u] = p;
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (h0 + u >= g) continue;
        const u64* v = s_key + (h0 + u) * r;
        int up = pos[u];
        if (up < r && v[up] == y)  // ties: the first key above y
          for (int step = top; step > 0; step >>= 1)
            if (up + step <= r && v[up + step - 1] <= y) up += step;
        j2 += (u64)(pos[u] + up);
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) j2 += __shfl_xor_sync(0xffffffffu, j2, o);
  if ((tid & 31) == 0) s_j2[tid >> 5] = j2;
  __syncthreads();
  if (tid >= 32) return;
  // group means of the finite realizations, summed in realization order: the
  // smallest L by lane 0, the largest by lane 1
  double mean = nan("");
  if (tid < 2) {
    const int g = (tid == 0) ? 0 : n_L - 1;
    const double* v = src + (int64_t)ord.group[g] * r;
    double t = 0.0;
    for (int k0 = 0; k0 < r; k0 += 8) {
      double x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = (k0 + u < r) ? v[k0 + u] : INFINITY;
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (order_key((u64)__double_as_longlong(x[u])) != kMissing) t = __dadd_rn(t, x[u]);
    }
    if (s_cnt[g] > 0) mean = __ddiv_rn(t, (double)s_cnt[g]);
  }
  const double mean_last = __shfl_sync(0xffffffffu, mean, 1);
  if (tid != 0) return;
  unsigned long long J2 = 0ull;
  for (int w = 0; w < kConvThreads / 32; ++w) J2 += s_j2[w];
  double N = 0.0, S2 = 0.0, S3 = 0.0;
  for (int g = 0; g < n_L; ++g) {
    const double n = (double)s_cnt[g];
    N = __dadd_rn(N, n);
    S2 = __dadd_rn(S2, __dmul_rn(n, n));
    S3 = __dadd_rn(S3, __dmul_rn(__dmul_rn(n, n), __dadd_rn(__dmul_rn(2.0, n), 3.0)));
  }
  const double J = 0.5 * (double)J2;  // exact: J2 < 2^53
  const double mean_j = __ddiv_rn(__dsub_rn(__dmul_rn(N, N), S2), 4.0);
  const double var = __ddiv_rn(
      __dsub_rn(__dmul_rn(__dmul_rn(N, N), __dadd_rn(__dmul_rn(2.0, N), 3.0)), S3), 72.0);
  ConvergenceRow o;
  o.jt = J;
  o.z = (var > 0.0) ? __ddiv_rn(__dsub_rn(J, mean_j), __dsqrt_rn(var)) : nan("");
  o.rho_first = mean;
  o.rho_last = mean_last;
  o.n_valid = (int32_t)N;
  o.converged = (o.z > z_crit && o.rho_last > o.rho_first && o.rho_last > 0.0) ? 1 : 0;
  out[row] = o;
}

}  // namespace

size_t convergence_smem(int32_t n_L, int32_t r) { return (size_t)n_L * (size_t)r * 8; }

cudaError_t convergence_prepare() {
  return cudaFuncSetAttribute(convergence_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)(kMaxConvValues * 8));
}

cudaError_t launch_convergence(const double* rho, int64_t n_rows, int32_t n_L, int32_t r,
                               const ConvOrder& ord, double z_crit, ConvergenceRow* out,
                               cudaStream_t s) {
  if (n_rows <= 0) return cudaSuccess;
  convergence_kernel<<<(unsigned)n_rows, kConvThreads, convergence_smem(n_L, r), s>>>(
      rho, n_L, r, ord, z_crit, out);
  return cudaGetLastError();
}

}  // namespace ccm
