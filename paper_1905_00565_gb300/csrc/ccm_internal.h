// Internal declarations shared by the CUDA kernels and the host runtime of the
// CCM library (not part of the public ABI, see include/ccm.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace ccm {

constexpr int kMaxE = 10;
constexpr int kSms = 152;  // a GB300's: launches are split for so many

// One library realization ("unit"): library variable j, E, tau, L, realization
// k of one job, with the targets it is cross-mapped to.  The library and the
// neighbour lists do not depend on the target, so all pairs (j, i) of a job
// that share j are computed from one neighbour search.
struct UnitDesc {
  int64_t series_off;   // element offset of the job's series block [V][n]
  int64_t lib_off;      // offset of this unit's library in the library buffer (units that read a
                        // table share one slot there: only the plain comparator lists them)
  int64_t bits_off;     // table_R > 0: this unit's membership bits, by position of the query order
                        // (consecutive units of one cell lie back to back)
  int64_t words_off;    // units read in groups: their membership words; -1: none
  int64_t part_off;     // first partial-sum slot: target t, tile q at part_off + t*n_tiles + q
  int64_t order_off;    // first entry of this unit's query order (per variable, E, tau)
  int64_t tgt_off;      // first TargetDesc of this unit
  int64_t table_off;    // distance indexing table of (j, E, tau), when table_R > 0
  int64_t st_off;       // the job's series by time, [n][st_stride]; -1: there is none
  uint64_t seed;        // library sampler seed of the job
  int32_t n;            // series length of the job
  int32_t j;            // library variable
  int32_t tau;
  int32_t L, k;
  int32_t n_m;          // manifold points = queries
  int32_t n_tiles;      // query tiles of the fused kernel
  int32_t n_targets;    // targets cross-mapped from this library (>= 1)
  int16_t E;
  int16_t table_R;      // > 0: neighbours read from the table (its row length, a multiple of 64)
  int32_t theiler;      // exclusion window W >= 0: candidates l of query m need |l - m| > W
  float wfloor;         // simplex weight floor f >= 0: u_i = max(u_i, f)
  int32_t st_stride;
};
static_assert(sizeof(UnitDesc) == 128, "no padding");
// Units with at least this many targets form their predictions with one lane
// per target (coalesced reads of the time-major series, where the plan has room
// for that copy); others, one thread per query and target after target.
constexpr int kLaneTargets = 12;
__host__ __device__ inline bool lane_per_target(const UnitDesc& u) {
  return u.n_targets >= kLaneTargets && u.st_off >= 0;
}

// One target of a unit: the pair (j, i) and where its outputs go.
struct TargetDesc {
  int64_t out_idx;      // index of this (pair, E, tau, L, k) in the rho buffer
  int64_t q_off;        // first query of this pair-realization in the debug predictions
  int64_t nbr_off;      // first entry in the debug neighbour lists
  int64_t lib_dbg_off;  // first entry in the debug libraries
  int64_t obs_tile;     // observed-value record of query tile 0 of (j, i, E, tau)
  int32_t i;            // target variable
  int32_t unit;         // the unit it belongs to
};

// Observed-value job: one per (job, library variable j, target i, E, tau).
// The observed values of a query tile (the target at the tile's manifold
// points) do not depend on L or the realization, so their tile mean, centred
// values and centred sum of squares are computed once per run and read by the
// epilogue of every realization of that (j, i, E, tau).  All values are scaled
// by the target series' power of two (moments.cuh).
struct ObsJob {
  int64_t series_off;   // element offset of the job's series block
  int64_t n;            // series length
  int64_t order_off;    // query order of (j, E, tau)
  int64_t obs_tile;     // first tile's ObsStat; the jobs' records are consecutive
  int64_t a_off;        // centred values: element of query 0 of tile 0
  int32_t a_step;       // 0: a tile's 256 values in obs_slot order; T > 0: query q of tile t at
                        // a_off + (256t + q)*T (the T targets of a query side by side)
  int32_t scale;        // index of the target series' scale
  int32_t i, E, tau, n_m, n_tiles;
  int32_t pad;
};
// A target series' power of two, and the smallest sum of squares at which a tile of
// its predictions may need a second look (moments.cuh): the smallest positive
// number, or 0 for a deep series, one with (nonzero) values below 2^-kDeepBits of its
// largest, where a sum of 0 does not show that all predictions are equal.
constexpr int kDeepBits = 90;
struct alignas(8) SeriesScale {
  float scale, least_b2;
};
// One tile of an observed target: mean(x), sum of (x_q - mean(x))^2 and the
// scale.  Beside it 256 float2 {h, l}, h + l = x_q - mean(x) to 48 bits (zero
// past the tile's end).
struct ObsStat {
  double mx, sxx;
  SeriesScale series;   // the series'
  float pad[2];
};
// Per-series preparation (one CTA of the order launch): the power of two that
// brings the series' largest magnitude into 2^kScaleBits times [1, 2) (less for
// series below 2^(kScaleBits - 127)), and, for jobs with units of kLaneTargets
// targets, the series' column of the time-major copy.
constexpr int kScaleBits = 50;
struct SeriesJob {
  int64_t off, n;       // the series
  int64_t st_off;       // element of (t = 0, this variable) in the time-major copy; -1: none
  int32_t st_stride;
  int32_t scale;        // where the scale goes
};

// One work item of the search kernels: query tiles of a unit, from `tile` on;
// the last item of a unit may hold fewer than its count says.
//   brute force: up to `count` tiles (brute_chunk)
//   table scan of units with one target (knn_scan.cu): (count >> 8) tiles of
//     count & 255 consecutive units, realizations of one (j, E, tau)
//   table walk of units with several targets: up to kTableChunk tiles
struct WorkItem {
  int32_t unit;
  int32_t tile;
  int32_t count;
};
constexpr int kBruteChunk = 8;         // query tiles per brute-force work item, at most
// Points of a staged library tile in the brute-force kernel: kTileBytes of
// packed coordinate pairs (padded to even E) and indices, whole warps of them.
constexpr int kTileBytes = 20 * 1024;
constexpr int brute_tile_points(int E) {
  return (kTileBytes / ((E + (E & 1)) * 8 + 8)) * 2 / 64 * 64;
}
// Query tiles per brute-force item, for libraries of L points in a launch of
// `tiles` tiles.  An item is the unit of balance, and a launch of few
// realizations has too few of eight tiles for the 152 SMs x 3 CTA slots (50
// realizations of N = 10^4, L = 1500: 250 items of 8 tiles 620 us, 2000 items
// 440 us).  A library that fits one staged tile is staged once per item (3-8 %
// of a tile's time), so there one item per slot is enough: with eight, 2400
// tiles of N = 1000 and L <= 200 took 1.5 % longer.  Longer libraries are
// staged for every tile anyway and are split to eight items per slot.
constexpr int64_t kBruteSlots = 3 * kSms;
inline int32_t brute_chunk(int64_t tiles, int64_t L, int E) {
  const int64_t c = tiles / (L <= brute_tile_points(E) ? kBruteSlots : 8 * kBruteSlots);
  return c < 1 ? 1 : c > kBruteChunk ? kBruteChunk : (int32_t)c;
}
constexpr int kScanGroup = 32;         // realizations per scan item: one lane each
constexpr int kScanChunk = 8;          // query tiles per scan item, at most
constexpr size_t kScanSmemMax = 112 * 1024;  // shared memory of a scan CTA: two fit an SM
// Membership words of a scan group: one per position of the query order, and
// zeros up to a whole number of 32 beyond the last (table rows are padded with
// position n_m).
__host__ __device__ constexpr int member_words(int n_m) { return (n_m + 32) / 32 * 32; }
// Shared memory of a scan CTA: 32 vectors of predictions (vec_slot order of 256; the
// odd stride spreads the 32 lanes' stores of one query over the banks) and the lanes'
// records of E+1 steps; then the membership words, while two CTAs still fit an SM
// (manifolds up to 18656 points for E = 1, 11744 for E = 10).
constexpr int kScanThreads = 512;
constexpr int kScanVec = 256 + 9;
__host__ __device__ constexpr size_t scan_fixed_smem(int E) {
  return 32 * kScanVec * 4 + (size_t)(E + 1) * kScanThreads * (4 + 2);
}
__host__ __device__ constexpr bool scan_words_in_smem(int E, int64_t n_m) {
  return n_m < 65536 &&
         scan_fixed_smem(E) + (size_t)member_words((int)n_m) * 4 <= kScanSmemMax;
}
// Realizations of an item of units with many targets that read a table: the
// weights and neighbours of a query tile wait in 160 KB of shared memory.
__host__ __device__ constexpr int lane_group(int E) {
  return 80 / (E + 1) < kScanGroup ? 80 / (E + 1) : kScanGroup;
}
constexpr size_t kGroupSmemMax = 224 * 1024;  // shared memory of its CTA: one an SM
// One scan group: `count` consecutive units from `unit` on.
struct MemberGroup {
  int32_t unit, count;
};

// Query order job: one per (job, library variable, E, tau).
struct OrderJob {
  int64_t series_off;   // element offset of the job's series block
  int64_t n;            // series length
  int64_t order_off;    // first entry of the order array of this combination
  int64_t scratch_off;  // manifolds above kOrderMaxSort: 2*n_m 64-bit keys of scratch
                        // from here (merge sort); -1: keep time order
  int32_t j, E, tau, n_m;
};
constexpr int kOrderMaxSort = 16384;   // manifolds up to this size are sorted in one pass

// Distance indexing table job: one per (job, library variable, E, tau) whose
// realizations read their neighbours from a table.
struct TableJob {
  int64_t series_off;   // element offset of the job's series block
  int64_t n;            // series length
  int64_t order_off;    // query order of this combination
  int64_t table_off;    // first entry: rank r of query position pos at table_off + pos*stride + r
  int32_t j, E, tau, n_m;
  int32_t R;            // entries per row; padded with position n_m to
  int32_t stride;       // a multiple of 64
  int64_t pts_off;      // the points in query order: [chunk of 32][E][32] floats
  int64_t box_off;      // chunk boxes [2E][32 * superchunks], superchunk boxes [2E][superchunks]
  int64_t sbox_off;
  int64_t least_off;    // smallest manifold index of every chunk, of every superchunk (int32)
  int64_t sample_off;   // every sample-th point, [E][n_m / sample]
  int32_t sample;       // (sample_stride)
  int32_t tv_i;         // >= 0: also store target variable tv_i's value at every entry's point
};
// The sample a row's threshold is read from: at least about 1000 points, and about
// eight of them at the distance aimed at (a third of the count either way, which
// the row's capacity takes).  With 24, short rows were sampled in full: three
// tables of N = 9000, E = 3, R = 32 1.34 ms, now 1.24; 8 of N = 10^5 36.5, now 35.5.
inline int32_t sample_stride(int64_t n_m, int64_t R) {
  int32_t s = 1;
  while (2 * s * 1024 <= n_m && 2 * s * 8 <= R + 32) s <<= 1;
  return s;
}
constexpr int kTableMaxR = 4096;       // entries per query row, at most
constexpr int kWalkMaxR = 2048;        // the same for variables with several targets
constexpr int kTableChunk = 8;         // query tiles per table work item (one bitmap each)
constexpr int kTableMaxNm = 1 << 20;   // longest manifold that gets a table (bitmap in smem)

// Sampler: one CTA per unit.
struct SamplerParams {
  const UnitDesc* units;
  const TargetDesc* targets;  // for the debug copies (lib_dbg_off per target)
  const int32_t* order;   // query orders (per variable, E, tau); libraries follow them
  int32_t* lib;           // library buffer (sum of L), each library in query order
  uint32_t* bits;         // membership bits of the units that read a table (no list is written)
  int32_t list_all;       // 1: list those too (at lib_off)
  int32_t window;         // > 0: list at most so many keys around the last member's
  int32_t* dbg_lib;       // optional: libraries in ascending m, once per target, in rho order
  int32_t* err;           // error flag (set, never cleared, by the kernels)
};

// Fused kNN + simplex + moments: persistent, one work item at a time.
struct KnnParams {
  const float* series;    // device series blocks
  const UnitDesc* units;
  const TargetDesc* targets;
  const WorkItem* items;
  int64_t n_items;
  const int32_t* lib;
  const int32_t* order;   // query order (manifold index per position)
  const uint32_t* bits;   // membership bits of the units that read a table
  const uint32_t* words;  // membership words of the scan groups
  const void* table;      // distance indexing tables (units with table_R > 0)
  const float* table_dist;  // every table entry's distance sqrt_hw(FP32 squared distance), same
                            // layout; table_pairs: float2 {distance, target value} per entry
  int32_t table_pairs;    // 1: the tables store (distance, target value) pairs (TableJob::tv_i)
  int32_t window;         // 1: some unit has an exclusion window
  int32_t table_u16;      // 1: uint16 entries (every manifold below 65536 points), 0: int32
  float4* partials;       // two float4 per (target, query tile): its sums (moments.cuh)
  const float2* obs;      // centred observations, 256 per record (TargetDesc::obs_tile)
  const ObsStat* obs_stat;  // one per record
  const float* st;        // time-major series of jobs with units of kLaneTargets targets
  uint32_t* item_counter; // dynamic scheduling counter (zeroed before each launch)
  int32_t* dbg_nbr;       // optional [sum N_m][E+1]
  float* dbg_xhat;        // optional [sum N_m]
  int32_t* err;
  unsigned long long* stats;  // optional search counters [kStatCount] (kStat*), nullptr: none
  int32_t lane_scratch;   // table kernel: where the lane-per-target scratch starts in shared memory
  int32_t prune;          // brute force: 0: the manifold keeps time order, nothing to exclude
  int32_t group_words;    // grouped table kernel: membership words in shared memory
  int32_t persistent;     // 1: CTAs pull items from item_counter; 0: item = blockIdx.x
  int32_t merge_at[kMaxE + 1];  // per E: merge pending candidates once a lane holds this many
  int32_t variant[kMaxE + 1];   // per E: kernel variant (0 narrow, 1 wide); same results
};

// Search counters, accumulated by the kernels when KnnParams::stats is set (a
// separately compiled counting variant; the results are the same).
enum : int {
  kStatBruteTiles = 0,   // query tiles searched by brute force
  kStatBruteQueries,     // their valid queries
  kStatPairsBegun,       // query-library pairs whose distance was begun (lanes x points)
  kStatPairsFull,        // pairs whose distance was completed over all E coordinates
  kStatPairsPruned,      // pairs skipped by the box test (lanes x points)
  kStatCandidates,       // candidates appended to the pending buffers
  kStatMergeSlots,       // lockstep insertion slots: per warp merge, 32 x its largest pending count
  kStatTableQueries,     // valid queries answered from a distance indexing table
  kStatTableEntries,     // table entries loaded (one walk may serve several realizations)
  kStatTableFallbacks,   // queries that scanned their library instead
  kStatCount = 16
};

// Defaults before tuning: merge trigger (pending candidates per lane) and variant.
constexpr int kDefaultMergeAt = 4;
constexpr int kDefaultVariant = 1;

// Hardware square root and reciprocal (sqrt.approx.f32, rcp.approx.f32:
// within about one ulp, subnormal inputs included).
__device__ __forceinline__ float sqrt_hw(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rcp_hw(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Simplex weight (paper Sect. 2.1) of a neighbour at distance d = sqrt_hw(d2)
// when the nearest is at distance d1 (> 0; inv_d1 = rcp_hw(d1)): u =
// exp(-d/d1), raised to the floor f.  d1 = 0 takes the limit: 1 for d = 0,
// else 0.  Shared by the fused kernels and the plain comparator so that all
// compute the same bits; FP32 with the hardware square root, reciprocal and
// exponential (relative error near 1e-7, far inside the 1e-5 the predictions
// are checked to).  The two cases separately, then together:
__device__ __forceinline__ float simplex_exp(float d, float inv_d1) {  // d1 > 0
  return __expf(-__fmul_rn(d, inv_d1));
}
__device__ __forceinline__ float simplex_limit(float d) {  // d1 = 0
  return (d == 0.f) ? 1.f : 0.f;
}
__device__ __forceinline__ float simplex_u_dist(float d, float d1, float inv_d1, float wfloor) {
  return fmaxf((d1 > 0.f) ? simplex_exp(d, inv_d1) : simplex_limit(d), wfloor);
}
__device__ __forceinline__ float simplex_u(float d2, float d1, float inv_d1, float wfloor) {
  return simplex_u_dist(sqrt_hw(d2), d1, inv_d1, wfloor);
}

// Where a launch goes.  chained: its CTAs may be set up while the kernel before
// it on the stream drains (launch.cuh).  Only for the direct launches of one
// job: inside a captured graph the gaps are short anyway (175 against 170 us for
// a single job), and set-up CTAs hold resources that other streams' kernels
// could use (a served burst: 7.3 against 7.0 ms).
struct LaunchStream {
  cudaStream_t s;
  bool chained;
  LaunchStream(cudaStream_t stream, bool chain = false) : s(stream), chained(chain) {}
};

// Error flag values written by kernels.
constexpr int32_t kErrBadUnit = 1;
constexpr int32_t kErrSampler = 2;
constexpr int32_t kErrTable = 4;

// Sampler (sampler.cu).
constexpr int kSamplerThreads = 256;
constexpr int kSamplerBitsMax = 1 << 20;  // membership bits in shared memory up to this N_m
cudaError_t sampler_prepare();
cudaError_t launch_sampler(const SamplerParams& p, int64_t first_unit, int64_t count,
                           int max_nm, LaunchStream s);
// Membership words of the scan groups from their units' bits.
cudaError_t launch_member_words(const UnitDesc* units, const MemberGroup* groups, int64_t n_groups,
                                int max_nm, const uint32_t* bits, uint32_t* words, LaunchStream s);

// Query order (order.cu).
cudaError_t order_prepare();
// inverse (optional): the position of every manifold index, same offsets.
// The same launch prepares the target series (SeriesJob).
cudaError_t launch_order(const float* series, const OrderJob* jobs, int64_t n_jobs, int max_nm,
                         int32_t* order, int32_t* inverse, unsigned long long* scratch,
                         const SeriesJob* series_jobs, int64_t n_series_jobs, SeriesScale* scales,
                         float* st, LaunchStream s);

// Distance indexing table (table.cu).
cudaError_t table_prepare();
// The jobs' points and boxes (all jobs of a run).
cudaError_t launch_table_points(const float* series, const TableJob* jobs, int64_t n_jobs,
                                int max_nm, const int32_t* order, float* points, LaunchStream s);
// One launch builds the tables of jobs[0..n_jobs), all of embedding dimension E
// (n_rows rows together).
cudaError_t launch_table_build(const float* series, const TableJob* jobs, int64_t n_jobs,
                               int64_t n_rows, int E, int max_nm, int max_R, const float* points,
                               const int32_t* order, const int32_t* inverse, void* table,
                               float* table_dist, int table_pairs, int table_u16, int32_t* err,
                               LaunchStream s);
// Its kernels (table_build.cu, compiled once per E).
template <int E>
struct TableKernels {
  static cudaError_t prepare();
  static cudaError_t launch(const float* series, const TableJob* jobs, int64_t n_jobs,
                            int64_t n_rows, int max_nm, int max_R, const float* points,
                            const int32_t* order, const int32_t* inverse, void* table,
                            float* table_dist, int pairs, int u16, int32_t* err, LaunchStream s);
};

// Search kernels of one E (knn_fused.cu, compiled once per E; each kernel keeps
// its registers for that E's lists).
template <int E>
struct KnnKernels {
  static cudaError_t prepare();
  static cudaError_t occupancy(int* ctas);
  static cudaError_t launch(const KnnParams& p, bool lanes, int grid, LaunchStream s);
  static cudaError_t prepare_table();
  static cudaError_t occupancy_table(int max_nm, bool lanes, int* ctas);
  static cudaError_t launch_table(const KnnParams& p, int max_nm, bool lanes, int grid,
                                  LaunchStream s);
  static cudaError_t prepare_group();
  static cudaError_t launch_group(const KnnParams& p, int max_nm, int grid, LaunchStream s);
  static cudaError_t prepare_scan();
  static cudaError_t launch_scan(const KnnParams& p, int max_nm, int grid, LaunchStream s);
};

// Their dispatch, and what surrounds the search (knn_dispatch.cu).
int knn_block_threads();
int knn_queries_per_thread();
cudaError_t knn_prepare();
cudaError_t knn_occupancy(int E, int* ctas_per_sm);
// lane_targets: the launch's units have kLaneTargets targets or more (a kernel
// of their own).
cudaError_t launch_knn(const KnnParams& p, int E, bool lane_targets, int grid, LaunchStream s);
// Observed-value records of every ObsJob (after the query order): one warp
// per tile, n_tiles tiles in all.
cudaError_t launch_obs(const float* series, const int32_t* order, const ObsJob* jobs,
                       int64_t n_jobs, int64_t n_tiles, const SeriesScale* scales, float2* obs,
                       ObsStat* obs_stat, LaunchStream s);
// rho of every target from its tiles' sums (after the search kernels).
cudaError_t launch_rho(const UnitDesc* units, const TargetDesc* targets, int64_t n_targets,
                       int max_tiles, const float4* partials, const ObsStat* obs_stat, double* rho,
                       LaunchStream s);
// Table path: same work items, neighbours read from the distance indexing table.
cudaError_t knn_table_prepare();
cudaError_t knn_table_occupancy(int max_nm, bool lane_targets, int* ctas_per_sm);
cudaError_t launch_knn_table(const KnnParams& p, int E, int max_nm, bool lane_targets, int grid,
                             LaunchStream s);
// Units with one target: grouped realizations (two CTAs per SM; knn_scan.cu).
cudaError_t knn_scan_prepare();
cudaError_t launch_knn_scan(const KnnParams& p, int E, int max_nm, int grid, LaunchStream s);

// Units with many targets: grouped realizations (one CTA per SM).
cudaError_t knn_group_prepare();
cudaError_t launch_knn_group(const KnnParams& p, int E, int max_nm, int grid, LaunchStream s);

// Sets the thread-local message returned by ccm_last_error() (runtime.cu).
void set_last_error(const char* msg);

// Plain comparator (plain.cu): one realization per call.
// Convergence decision (one CTA per (pair, E, tau) row of the rho grid).
constexpr int kMaxConvGroups = 64;      // L values per row, at most
constexpr int kMaxConvValues = 24576;   // n_L * r per row, at most (shared memory)
struct ConvOrder {
  int32_t group[kMaxConvGroups];        // L-axis index of the g-th smallest L
};
struct ConvergenceRow {                 // same layout as ccm_convergence_t
  double rho_first, rho_last, jt, z;
  int32_t n_valid, converged;
};
cudaError_t convergence_prepare();
cudaError_t launch_convergence(const double* rho, int64_t n_rows, int32_t n_L, int32_t r,
                               const ConvOrder& ord, double z_crit, ConvergenceRow* out,
                               cudaStream_t s);

cudaError_t launch_plain_unit(const float* series, const UnitDesc* unit_dev, const UnitDesc& unit,
                              const TargetDesc* target_dev, const int32_t* lib,
                              float* xhat_scratch, double* rho_out, cudaStream_t s);

}  // namespace ccm
