// Host runtime of the CCM library: the C ABI of include/ccm.h.
//
//  * context: device, device-memory budget, one-time kernel set-up, serving
//    thread;
//  * plan: validated copy of a problem, its realizations ("units") in output
//    order, the work list of (unit, query tile) items sorted by decreasing
//    cost, and one device arena for series, libraries, partial moments and rho;
//  * run: query orders, tables, sampler, one search launch per E and kind of
//    unit, rho; captured once into a CUDA graph and replayed;
//  * plain comparator: one launch sequence per realization;
//  * serving: queued jobs are admitted while their footprints fit the free
//    budget, admitted jobs are batched into shared launches on a pool of
//    streams, and results are copied back per job.
#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <sys/stat.h>
#include <cstring>
#include <deque>
#include <list>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <tuple>
#include <vector>

#include "ccm.h"
#include "ccm_internal.h"

using namespace ccm;

namespace {

thread_local std::string t_err;

ccm_status fail(ccm_status st, const std::string& msg) {
  t_err = msg;
  return st;
}

#define CCM_CUDA(call)                                                                   \
  do {                                                                                   \
    const cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess)                                                               \
      return fail(CCM_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_));        \
  } while (0)

double now_s() {
  using namespace std::chrono;
  return duration<double>(steady_clock::now().time_since_epoch()).count();
}

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---------------------------------------------------------------- problem ---
struct ProblemCopy {
  int32_t V = 0;
  int64_t n = 0;
  std::vector<int32_t> pairs, E, tau;
  std::vector<int64_t> L;
  int32_t r = 0;
  uint64_t seed = 0;
  uint32_t flags = 0;
  int32_t theiler = 0;
  float weight_floor = 0.f;

  int64_t n_units() const {
    return (int64_t)(pairs.size() / 2) * (int64_t)E.size() * (int64_t)tau.size() *
           (int64_t)L.size() * r;
  }
};

ccm_status copy_problem(const ccm_problem* p, ProblemCopy* pc) {
  if (!p) return fail(CCM_EINVAL, "problem is NULL");
  if (p->n_series < 2) return fail(CCM_EINVAL, "n_series must be >= 2");
  if (p->n < 3 || p->n > 0x7fffffff) return fail(CCM_EINVAL, "series length out of range");
  if (p->n_pairs < 1 || !p->pairs) return fail(CCM_EINVAL, "no pairs");
  if (p->n_E < 1 || !p->E || p->n_tau < 1 || !p->tau || p->n_L < 1 || !p->L)
    return fail(CCM_EINVAL, "empty E, tau or L grid");
  if (p->r < 1) return fail(CCM_EINVAL, "r must be >= 1");
  pc->V = p->n_series;
  pc->n = p->n;
  pc->pairs.assign(p->pairs, p->pairs + 2 * (size_t)p->n_pairs);
  pc->E.assign(p->E, p->E + p->n_E);
  pc->tau.assign(p->tau, p->tau + p->n_tau);
  pc->L.assign(p->L, p->L + p->n_L);
  pc->r = p->r;
  pc->seed = p->seed;
  pc->flags = p->flags;
  if (p->flags & ~(uint32_t)(CCM_INPUT_ON_DEVICE | CCM_OUTPUT_ON_DEVICE | CCM_NO_AUTOTUNE |
                             CCM_NO_TABLE | CCM_SEARCH_STATS))
    return fail(CCM_EINVAL, "unknown flag bits");
  pc->theiler = p->theiler;
  pc->weight_floor = p->weight_floor;
  if (p->theiler < 0) return fail(CCM_EINVAL, "theiler window must be >= 0");
  if (!std::isfinite(p->weight_floor) || p->weight_floor < 0.f)
    return fail(CCM_EINVAL, "weight_floor must be finite and >= 0");
  for (int32_t q = 0; q < p->n_pairs; ++q) {
    const int32_t j = pc->pairs[2 * q], i = pc->pairs[2 * q + 1];
    if (j < 0 || j >= pc->V || i < 0 || i >= pc->V || i == j)
      return fail(CCM_EINVAL, "pair " + std::to_string(q) + " is invalid (need 0<=i,j<V, i!=j)");
  }
  {
    // the interface's limit: (pairs sharing a library variable) x (query tiles) in 32 bits
    std::map<int32_t, int64_t> targets_of;
    int64_t most = 0;
    for (int32_t q = 0; q < p->n_pairs; ++q) most = std::max(most, ++targets_of[pc->pairs[2 * q]]);
    if (most * ((pc->n + 255) / 256) > 0x7fffffff)
      return fail(CCM_EINVAL, "targets of one library variable x query tiles exceed 2^31 - 1");
  }
  for (int32_t E : pc->E)
    if (E < 1 || E > kMaxE) return fail(CCM_EINVAL, "E must be in 1..10");
  for (int32_t t : pc->tau)
    if (t < 1) return fail(CCM_EINVAL, "tau must be >= 1");
  for (int32_t E : pc->E)
    for (int32_t t : pc->tau) {
      const int64_t n_m = pc->n - (int64_t)(E - 1) * t;
      for (int64_t L : pc->L) {
        if (L < E + 2 || L > n_m)
          return fail(CCM_EINVAL, "L=" + std::to_string(L) + " outside [E+2, N_m] for E=" +
                                      std::to_string(E) + ", tau=" + std::to_string(t));
        if (L < (int64_t)E + 2 + 2 * (int64_t)pc->theiler)
          return fail(CCM_EINVAL, "L=" + std::to_string(L) + " < E+2+2W for E=" +
                                      std::to_string(E) + ", W=" + std::to_string(pc->theiler));
      }
    }
  if ((double)pc->n_units() > 2.0e9) return fail(CCM_EINVAL, "too many realizations");
  return CCM_OK;
}

bool all_finite(const float* x, size_t count) {
  for (size_t q = 0; q < count; ++q)
    if (!std::isfinite(x[q])) return false;
  return true;
}

// ------------------------------------------------------------- unit lists ---
// The work items of one search launch: one E, and units of one, few or many
// targets (a kernel each; brute force: one and few share theirs), or of many
// whose realizations read their table in groups.
enum class Targets : int32_t { kOne, kFew, kMany, kGrouped };
struct ItemGroup {
  int32_t E;
  Targets targets;
  int64_t first, count;
  int32_t max_nm;  // longest manifold of its units: the launch's shared memory follows it
};

struct UnitList {
  std::vector<UnitDesc> units;        // library realizations
  std::vector<TargetDesc> targets;    // their targets (one per output rho)
  std::vector<WorkItem> items;        // brute-force items, grouped by E (see sort_items)
  std::vector<double> item_cost;
  std::vector<ItemGroup> groups;      // brute-force launches, in stream order
  std::vector<ItemGroup> groups_table;  // the same for the table items
  std::vector<OrderJob> orders;       // one per (job, library variable, E, tau)
  std::vector<ObsJob> obs_jobs;       // one per (job, library variable, target, E, tau)
  int64_t obs_total = 0;              // observed-value tile records
  std::vector<SeriesJob> series_jobs; // one per (job, target variable)
  int64_t st_total = 0;               // elements of the time-major series copies
  bool window = false;                // some unit has an exclusion window
  bool lane_targets = false;          // some unit has kLaneTargets targets
  std::vector<TableJob> tables;       // distance indexing tables to build
  std::vector<WorkItem> items_table;  // work items of units that read a table
  std::vector<MemberGroup> member_groups;  // scan groups (units of one target or many)
  int64_t bits_total = 0, words_total = 0;  // their membership bits and words
  int64_t lib_scratch = 0;            // longest library of the units that read a table
  std::vector<double> item_cost_table;
  int64_t lib_total = 0, part_total = 0, order_total = 0, table_total = 0;
  int64_t points_total = 0;           // floats: the tables' points and boxes
  int64_t order_scratch_total = 0;    // 64-bit keys for sorting manifolds above kOrderMaxSort
  // Table jobs are sorted by (size class, E) (sort_items) and built one launch
  // per size class (the power of two at or above R) and E: a launch's shared
  // memory follows its own longest row and its registers its E.
  static int table_rcap(int R) {
    int rc = 32;
    while (rc < R) rc <<= 1;
    return rc;
  }
  int table_groups() const {
    int g = 0;
    for (size_t q = 0; q < tables.size(); ++q)
      if (q == 0 || table_rcap(tables[q].R) != table_rcap(tables[q - 1].R) ||
          tables[q].E != tables[q - 1].E)
        ++g;
    return g;
  }
  double brute_flops = 0.0;           // 3E per pair of the units searched by brute force
  double brute_pairs = 0.0;           // query-library pairs of those units
  int64_t search_queries = 0;         // N_m summed over the units
  int64_t table_queries = 0;          // N_m summed over the units that read a table
  int32_t sampler_window = 0;         // CCM_SAMPLER_WINDOW
  bool table_tv = false;              // some table stores its target's values (TableJob::tv_i)
  Targets targets_of(const WorkItem& w) const {
    const UnitDesc& u = units[(size_t)w.unit];
    if (lane_per_target(u))
      return u.table_R > 0 && u.words_off >= 0 ? Targets::kGrouped : Targets::kMany;
    return u.table_R > 0 && u.n_targets == 1 ? Targets::kOne : Targets::kFew;
  }
  // The launches of a sorted item list.
  std::vector<ItemGroup> group_items(const std::vector<WorkItem>& list) const {
    std::vector<ItemGroup> g;
    for (size_t q = 0; q < list.size(); ++q) {
      const int32_t E = units[(size_t)list[q].unit].E;
      if (g.empty() || g.back().E != E || g.back().targets != targets_of(list[q]))
        g.push_back(ItemGroup{E, targets_of(list[q]), (int64_t)q, 0, 0});
      ++g.back().count;
      g.back().max_nm = std::max(g.back().max_nm, units[(size_t)list[q].unit].n_m);
    }
    return g;
  }
  int table_u16() const { return max_nm < 65536 ? 1 : 0; }
  size_t table_elem() const { return table_u16() ? 2 : 4; }
  int64_t n_rho = 0, q_total = 0, nbr_total = 0, lib_dbg_total = 0;  // per output realization
  int emin = kMaxE + 1, emax = 0, max_nm = 0;
  int table_max_nm = 0;               // longest manifold of the units that read a table
  double pairs = 0.0, flops = 0.0;    // neighbour-search work actually done
};

// Table tunables: the crossover constant c, the floor and the largest
// manifold-to-library ratio of table_min_L, and a factor s on the row length
// (see below).  The environment variables CCM_TABLE_CROSSOVER, CCM_TABLE_FLOOR,
// CCM_TABLE_MAX_RATIO and CCM_TABLE_SAFETY replace the defaults (read at each
// ccm_plan; tuning and measurement only); any of the first three leaves the
// decision to table_min_L.
struct TableTuning {
  double crossover, floor, max_ratio, safety;
  bool fixed;  // some threshold was given: the general rule alone decides
};
TableTuning read_table_tuning() {
  TableTuning r{20.0, 256.0, 40.0, 1.0, false};
  r.fixed = getenv("CCM_TABLE_CROSSOVER") || getenv("CCM_TABLE_FLOOR") || getenv("CCM_TABLE_MAX_RATIO");
  if (const char* e = getenv("CCM_TABLE_CROSSOVER")) r.crossover = std::max(0.0, atof(e));
  if (const char* e = getenv("CCM_TABLE_FLOOR")) r.floor = std::max(16.0, atof(e));
  if (const char* e = getenv("CCM_TABLE_MAX_RATIO")) r.max_ratio = std::max(1.0, atof(e));
  if (const char* e = getenv("CCM_TABLE_SAFETY")) r.safety = std::max(0.01, atof(e));
  return r;
}

// Smallest L whose realizations read a distance indexing table.  A table
// walk visits about (E+1)*N_m/L row entries per query; brute force (with chunk
// pruning) costs about L distance evaluations of E coordinates per query, far
// fewer at small E, where pruning skips most chunks.  Measured on GB300: on
// the N_m = 10^4 sweep (the table build included) c = 20 and a floor of 256
// are fastest, L ~ sqrt(c*N_m/(E+1)) being where a grouped table walk
// overtakes the selection-bound brute force of small libraries; on the
// N = 10^5 series (E = 3..6) brute force at L = 1000 beats walks of
// (E+1)*100 entries, so libraries below N_m/max_ratio (40) points stay with
// brute force.  The last term keeps the row length (table_row_length) within
// max_R.  (Measured with a walk per query and realization, which variables with
// two to eleven targets still take.  With many, whose walks serve a group of
// realizations, a lower floor gains nothing: 64 variables, N = 5000, L from 100:
// 56.3, 56.7, 59.0 ms a run with a floor of 256, 150, 90.)
double table_min_L(int32_t E, int64_t n_m, int max_R, const TableTuning& t) {
  return std::max({t.floor, std::ceil(std::sqrt(t.crossover * (double)n_m / (double)(E + 1))),
                   std::ceil((double)n_m / t.max_ratio),
                   std::ceil(t.safety * 2.8 * (E + 2) * (double)n_m / (double)max_R)});
}

// Row length R of a table whose smallest L is lmin.  A query of a realization
// with L = lmin finds a Poisson(lambda = R*lmin/N_m) number of its library's
// points among its R entries (the library is a uniform sample); with fewer
// than E+1 it scans its whole library instead, about lmin distance
// evaluations.  lambda is the smallest multiple of 1/4 for which that happens
// with probability at most 1/(10*lmin), so the misses cost at most about 0.1
// distance evaluations a query (times the safety factor s on lambda), and from
// lmin = 300 on still more rarely in proportion: there a miss's scan lasts longer
// than the tile that waits for it (two variables of N = 10^5: rows 5 % longer,
// scan 36 -> 29 ms).  2W more entries cover the points the exclusion window
// removes.
int64_t table_row_length(int32_t E, int64_t n_m, int64_t lmin, int32_t theiler, double safety) {
  const double eps = 1.0 / (10.0 * (double)lmin * std::max(1.0, (double)lmin / 300.0));
  double lambda = (double)(E + 1);
  for (;; lambda += 0.25) {
    double term = std::exp(-lambda), tail = term;  // P(X <= E), X ~ Poisson(lambda)
    for (int i = 1; i <= E; ++i) {
      term *= lambda / i;
      tail += term;
    }
    if (tail <= eps) break;
  }
  return (int64_t)std::ceil(safety * lambda * (double)n_m / (double)lmin) + 2 * (int64_t)theiler;
}

// Entries per row and their row stride (rows are padded to 64) of a table for
// libraries from lmin on: from the n_m - 1 points other than the query.
int64_t table_row_entries(int32_t E, int64_t n_m, int64_t lmin, int32_t theiler, double safety,
                          int max_R) {
  const int64_t R = table_row_length(E, n_m, lmin, theiler, safety);
  return std::min<int64_t>(std::min<int64_t>((R + 31) / 32 * 32, max_R), n_m - 1);
}

// Estimated picoseconds on one GB300: brute-force search of a query of one
// realization; table scan of it (W = ranks walked until the slowest of 32
// realizations has its E+1); table row of R entries.  Fitted to measurements
// at N = 1000..40000, E in {1, 3, 6, 10}, L = 20..1000 (e.g. N = 10^4, E = 6:
// brute force 140 / 265 / 472 ps at L = 100 / 400 / 1000, scan 87 / 42 / 26 ps,
// rows 58 / 22 / 15 ns), within a third of them.
double brute_ps(int32_t E, double L) {
  return 20.0 + 7.0 * E + (0.5 + 0.044 * E * E) * std::pow(L, 0.75);
}
double scan_ps(int32_t E, double n_m, double L) {
  const double W = (E + 1 + 2.3 * std::sqrt(E + 1.0)) * n_m / L;
  const bool in_smem = scan_words_in_smem(E, (int64_t)n_m);
  return 12.0 + 1.5 * E + 0.055 * W + (in_smem ? 0.0 : 15.0 + 0.03 * W);
}
double row_ps(int32_t E, double n_m, double R) {
  return 1e3 * (3.0 + 1.2 * E + 0.03 * R + 1.5e-4 * n_m);
}

// Smallest tabled L of a library variable with one target: that of the general
// rule (`base`; -1: no table), or the smaller one of the grid at which the
// brute-force searches it saves outweigh the scans and the longer rows by
// the estimates above (a table that the general rule does not build also costs
// about 10 us of launches).  Sweep of N = 10^4 (L = 100..9000, r = 250): every
// L tabled 172 ms a run, the general rule's 240 ms; two variables of N = 10^5
// (L from 1000): 106 against 120 ms.
int64_t cheapest_table_L(const ProblemCopy& pc, int32_t E, int64_t n_m, int64_t base, int max_R,
                         double safety) {
  auto cost = [&](int64_t lmin) {
    double c = 0.0;
    if (lmin >= 0) {
      c += row_ps(E, (double)n_m, (double)table_row_entries(E, n_m, lmin, pc.theiler, safety, max_R));
      if (base < 0) c += 10e6 / (double)n_m;
    }
    for (int64_t L : pc.L)
      c += pc.r * (lmin >= 0 && L >= lmin ? scan_ps(E, (double)n_m, (double)L) : brute_ps(E, (double)L));
    return c;
  };
  int64_t best = base;
  double least = cost(base);
  for (int64_t L : pc.L) {
    if (base >= 0 && L >= base) continue;
    // rows this long would not fit: too many queries would miss
    if (table_row_length(E, n_m, L, pc.theiler, safety) > max_R && n_m - 1 > max_R) continue;
    const double c = cost(L);
    if (c < least) {
      least = c;
      best = L;
    }
  }
  return best;
}

// Append the units of one problem.  Offsets: series block, first rho index.
// Pairs that share a library variable j share one library and one neighbour
// search per (E, tau, L, k); each pair becomes a target of that unit.
// room: what else the plan may hold.
struct Room {
  double table_bytes;  // distance indexing tables, at most
  bool time_major;     // the copy of the series that variables of many targets read
};
void append_units(const ProblemCopy& pc, int64_t series_off, int64_t out_base, UnitList* ul,
                  const Room& room) {
  const double table_cap_bytes = room.table_bytes;
  if (const char* e = getenv("CCM_SAMPLER_WINDOW")) ul->sampler_window = std::max(0, atoi(e));
  const int tileq = knn_block_threads() * knn_queries_per_thread();
  const int64_t nP = (int64_t)pc.pairs.size() / 2;
  const int64_t nE = (int64_t)pc.E.size(), nT = (int64_t)pc.tau.size(), nL = (int64_t)pc.L.size();
  const int64_t per_pair = nE * nT * nL * pc.r;
  // debug offsets of every output realization, in rho order
  std::vector<int64_t> q_off((size_t)(nP * per_pair)), nbr_off(q_off.size()), lib_off(q_off.size());
  {
    int64_t o = 0;
    for (int64_t p = 0; p < nP; ++p)
      for (int32_t E : pc.E)
        for (int32_t tau : pc.tau)
          for (int64_t L : pc.L)
            for (int32_t k = 0; k < pc.r; ++k, ++o) {
              const int64_t n_m = pc.n - (int64_t)(E - 1) * tau;
              q_off[(size_t)o] = ul->q_total;
              nbr_off[(size_t)o] = ul->nbr_total;
              lib_off[(size_t)o] = ul->lib_dbg_total;
              ul->q_total += n_m;
              ul->nbr_total += n_m * (E + 1);
              ul->lib_dbg_total += L;
            }
    ul->n_rho += o;
  }
  // library variables in order of first appearance, with their pairs
  std::vector<int32_t> lib_vars;
  std::map<int32_t, std::vector<int64_t>> pairs_of;
  for (int64_t p = 0; p < nP; ++p) {
    const int32_t j = pc.pairs[2 * p];
    if (!pairs_of.count(j)) lib_vars.push_back(j);
    pairs_of[j].push_back(p);
  }
  std::map<std::tuple<int32_t, int32_t, int32_t>, int64_t> combo;  // (j, E, tau) -> order_off
  for (int32_t j : lib_vars)
    for (int32_t E : pc.E)
      for (int32_t tau : pc.tau) {
        OrderJob oj;
        std::memset(&oj, 0, sizeof(oj));
        oj.series_off = series_off;
        oj.n = pc.n;
        oj.order_off = ul->order_total;
        oj.scratch_off = -1;
        oj.j = j;
        oj.E = E;
        oj.tau = tau;
        oj.n_m = (int32_t)(pc.n - (int64_t)(E - 1) * tau);
        combo[std::make_tuple(j, E, tau)] = oj.order_off;
        ul->order_total += oj.n_m;
        if (oj.n_m > kOrderMaxSort) {
          oj.scratch_off = ul->order_scratch_total;
          ul->order_scratch_total += 2 * (int64_t)oj.n_m;
        }
        ul->orders.push_back(oj);
      }
  // Target series: their scales and, when some library variable has many
  // targets, the time-major copy of the whole series block.
  bool lanes = false;
  auto many = [&](const std::vector<int64_t>& tp) {
    return room.time_major && tp.size() >= (size_t)kLaneTargets;
  };
  for (int32_t j : lib_vars) lanes |= many(pairs_of[j]);
  ul->lane_targets |= lanes;
  ul->window |= pc.theiler > 0;
  const int64_t st_off = lanes ? ul->st_total : -1;
  const int32_t st_stride = (pc.V + 31) / 32 * 32;
  if (lanes) ul->st_total += pc.n * st_stride;
  std::vector<int32_t> scale_of((size_t)pc.V, -1);
  for (int64_t p = 0; p < nP; ++p) {
    const int32_t i = pc.pairs[2 * p + 1];
    if (scale_of[(size_t)i] >= 0) continue;
    SeriesJob sj;
    std::memset(&sj, 0, sizeof(sj));
    sj.off = series_off + (int64_t)i * pc.n;
    sj.n = pc.n;
    sj.st_off = lanes ? st_off + i : -1;
    sj.st_stride = st_stride;
    sj.scale = scale_of[(size_t)i] = (int32_t)ul->series_jobs.size();
    ul->series_jobs.push_back(sj);
  }
  // Observed-value records per (j, E, tau) and target, shared by every L and k:
  // the targets of one (j, E, tau) lie side by side.
  std::map<std::tuple<int32_t, int32_t, int32_t>, int64_t> obs_of;  // first target's first record
  for (int32_t j : lib_vars)
    for (int32_t E : pc.E)
      for (int32_t tau : pc.tau) {
        const auto key = std::make_tuple(j, E, tau);
        if (!obs_of.emplace(key, ul->obs_total).second) continue;
        const int64_t base = ul->obs_total;
        const std::vector<int64_t>& tp = pairs_of[j];
        for (size_t t = 0; t < tp.size(); ++t) {
          ObsJob ob;
          std::memset(&ob, 0, sizeof(ob));
          ob.series_off = series_off;
          ob.n = pc.n;
          ob.order_off = combo[key];
          ob.obs_tile = ul->obs_total;
          ob.i = pc.pairs[2 * tp[t] + 1];
          ob.scale = scale_of[(size_t)ob.i];
          ob.E = E;
          ob.tau = tau;
          ob.n_m = (int32_t)(pc.n - (int64_t)(E - 1) * tau);
          ob.n_tiles = (ob.n_m + tileq - 1) / tileq;
          const bool side = many(tp);
          ob.a_step = side ? (int32_t)tp.size() : 0;
          ob.a_off = side ? base * tileq + (int64_t)t : ob.obs_tile * tileq;
          ul->obs_total += ob.n_tiles;
          ul->obs_jobs.push_back(ob);
        }
      }
  // Distance indexing tables (unless CCM_NO_TABLE): per (j, E, tau),
  // realizations from a smallest L on read their neighbours from a table of
  // the R nearest points of every query (R from table_row_length at that L).
  // The general rule takes L >= table_min_L and builds a table only when the
  // realizations that use it would otherwise scan at least 8*N_m library
  // points in total; for variables with one target, whose scan serves 32
  // realizations a walk, cheapest_table_L may go lower.  The plan's tables stay
  // within table_cap_bytes; the realizations of a (j, E, tau) without a table
  // use brute force.
  struct TableOf {
    int64_t off, lmin;
    int32_t stride;
  };
  std::map<std::tuple<int32_t, int32_t, int32_t>, TableOf> table_of;
  // The safety factor trades table memory and build time against how often a
  // query falls back to scanning its library.
  const TableTuning tt = read_table_tuning();
  const double safety = tt.safety;
  double table_bytes = 0.0;
  if (!(pc.flags & CCM_NO_TABLE)) {
    for (int32_t j : lib_vars)
      for (int32_t E : pc.E)
        for (int32_t tau : pc.tau) {
          const int64_t n_m = pc.n - (int64_t)(E - 1) * tau;
          if (n_m > kTableMaxNm) continue;
          const bool tv = pairs_of[j].size() == 1;  // the target's values stand in the rows
          const int max_R = tv ? kTableMaxR : kWalkMaxR;
          const double ls = table_min_L(E, n_m, kWalkMaxR, tt);
          int64_t base = -1;
          double lsum = 0.0;
          for (int64_t L : pc.L)
            if ((double)L >= ls) {
              base = (base < 0) ? L : std::min(base, L);
              lsum += (double)L * pc.r;
            }
          if (lsum < 8.0 * (double)n_m) base = -1;
          int64_t lmin = base;
          if (tv && !tt.fixed) lmin = cheapest_table_L(pc, E, n_m, base, max_R, safety);
          int64_t R = 0, stride = 0;
          double bytes = 0.0;
          auto size = [&]() {  // positions (2 or 4 bytes), distances, values
            R = table_row_entries(E, n_m, lmin, pc.theiler, safety, max_R);
            stride = (R + 63) / 64 * 64;
            bytes = (double)n_m * (double)stride * ((n_m < 65536 ? 2.0 : 4.0) + 4.0 + (tv ? 4.0 : 0.0));
          };
          if (lmin >= 0) size();
          if (lmin != base && table_bytes + bytes > table_cap_bytes) {
            lmin = base;  // too long for the cap: the general rule's
            if (lmin >= 0) size();
          }
          if (lmin < 0 || table_bytes + bytes > table_cap_bytes) continue;
          table_bytes += bytes;
          TableJob tj;
          std::memset(&tj, 0, sizeof(tj));
          tj.series_off = series_off;
          tj.n = pc.n;
          tj.order_off = combo[std::make_tuple(j, E, tau)];
          tj.table_off = ul->table_total;
          tj.j = j;
          tj.E = E;
          tj.tau = tau;
          tj.n_m = (int32_t)n_m;
          tj.R = (int32_t)R;
          tj.stride = (int32_t)stride;
          const int64_t chunks = (n_m + 31) / 32, supers = (chunks + 31) / 32;
          tj.pts_off = ul->points_total;
          tj.box_off = tj.pts_off + chunks * 32 * E;
          tj.sbox_off = tj.box_off + 2 * E * supers * 32;
          tj.sample = sample_stride(n_m, R);
          tj.least_off = tj.sbox_off + 2 * E * supers;
          tj.sample_off = tj.least_off + supers * 33;
          ul->points_total = (tj.sample_off + n_m / tj.sample * E + 63) / 64 * 64;
          tj.tv_i = tv ? pc.pairs[2 * pairs_of[j][0] + 1] : -1;
          if (tv) ul->table_tv = true;
          table_of[std::make_tuple(j, E, tau)] = TableOf{tj.table_off, lmin, tj.stride};
          ul->table_total += n_m * stride;
          ul->tables.push_back(tj);
        }
  }
  // Query tiles per brute-force and scan item, from the tiles of each E's launch.
  std::map<int32_t, int64_t> brute_tiles, scan_tiles, many_tiles;
  for (int32_t j : lib_vars)
    for (int32_t E : pc.E)
      for (int32_t tau : pc.tau) {
        const int64_t n_m = pc.n - (int64_t)(E - 1) * tau;
        const auto tab = table_of.find(std::make_tuple(j, E, tau));
        int64_t tabled = 0;
        for (int64_t L : pc.L) {
          if (tab == table_of.end() || L < tab->second.lmin)
            brute_tiles[E] += (n_m + tileq - 1) / tileq * pc.r;
          else
            tabled += pc.r;
        }
        if (many(pairs_of[j]))
          many_tiles[E] += (n_m + tileq - 1) / tileq * tabled;
        scan_tiles[E] += (n_m + tileq - 1) / tileq * ((tabled + kScanGroup - 1) / kScanGroup);
      }
  for (int32_t j : lib_vars) {
    const std::vector<int64_t>& tp = pairs_of[j];
    for (int64_t e = 0; e < nE; ++e)
      for (int64_t t = 0; t < nT; ++t) {
        const int32_t E = pc.E[(size_t)e], tau = pc.tau[(size_t)t];
        const size_t first_unit = ul->units.size();
        // Realizations per group of a variable with many targets: as many as
        // leave the launch two items per CTA.  The groups lose to a walk per
        // realization only where a launch is too small to fill them: 20
        // variables of N = 2000, r = 10, L = 1900 (one wave of items) 0.121 ms
        // against 0.114; 24 of 3000, r = 25, L = 500 .. 1900 0.76 against 1.07;
        // 32 of 3000, r = 20, L = 2800 0.33 against 0.39; 40 of 4000, r = 12, E = 8
        // 1.55 against 1.68.  Their byte offsets have 32 bits.
        const int32_t lanes_group =
            many(tp) && (uint64_t)pc.n * (uint64_t)st_stride * 4 < 1ull << 32
                ? (int32_t)std::min<int64_t>(many_tiles[E] / (2 * kSms), lane_group(E))
                : 0;
        const bool grouped = tp.size() == 1 || lanes_group >= std::min(8, lane_group(E));
        for (int64_t l = 0; l < nL; ++l) {
          const int64_t L = pc.L[(size_t)l];
          const int32_t chunk = brute_chunk(brute_tiles[E], L, E);
          for (int32_t k = 0; k < pc.r; ++k) {
            UnitDesc u;
            std::memset(&u, 0, sizeof(u));
            u.series_off = series_off;
            u.n = (int32_t)pc.n;
            u.j = j;
            u.E = (int16_t)E;
            u.tau = tau;
            u.L = (int32_t)L;
            u.k = k;
            u.seed = pc.seed;
            u.n_m = (int32_t)(pc.n - (int64_t)(E - 1) * tau);
            u.n_tiles = (u.n_m + tileq - 1) / tileq;
            u.n_targets = (int32_t)tp.size();
            u.theiler = pc.theiler;
            u.wfloor = pc.weight_floor;
            u.lib_off = ul->lib_total;
            u.part_off = ul->part_total;
            u.words_off = -1;
            u.st_off = st_off;
            u.st_stride = st_stride;
            u.order_off = combo[std::make_tuple(j, E, tau)];
            u.tgt_off = (int64_t)ul->targets.size();
            int64_t obs_tile = obs_of[std::make_tuple(j, E, tau)];
            for (int64_t p : tp) {
              const int64_t o = (((p * nE + e) * nT + t) * nL + l) * pc.r + k;  // rho order
              TargetDesc tg;
              std::memset(&tg, 0, sizeof(tg));
              tg.out_idx = out_base + o;
              tg.q_off = q_off[(size_t)o];
              tg.nbr_off = nbr_off[(size_t)o];
              tg.lib_dbg_off = lib_off[(size_t)o];
              tg.i = pc.pairs[2 * p + 1];
              tg.obs_tile = obs_tile;
              tg.unit = (int32_t)ul->units.size();
              obs_tile += u.n_tiles;
              ul->targets.push_back(tg);
            }
            const auto tab = table_of.find(std::make_tuple(j, E, tau));
            if (tab != table_of.end() && L >= tab->second.lmin) {
              u.table_off = tab->second.off;
              u.table_R = (int16_t)tab->second.stride;
              u.bits_off = ul->bits_total;
              ul->bits_total += (u.n_m + 31) / 32;
              ul->lib_scratch = std::max(ul->lib_scratch, L);
              ul->table_max_nm = std::max(ul->table_max_nm, u.n_m);
            }
            const int32_t uidx = (int32_t)ul->units.size();
            // the others get their items below, in groups
            const bool owns_items = !(u.table_R > 0 && grouped);
            for (int32_t q = 0; q < u.n_tiles && owns_items; ++q) {
              const int64_t nq = std::min<int64_t>(tileq, u.n_m - (int64_t)q * tileq);
              if (u.table_R > 0) {
                // one item per kTableChunk tiles: one copy of the membership
                // bits, then per tile one walk of each row and the epilogue
                if (q % kTableChunk == 0) {
                  ul->items_table.push_back(WorkItem{uidx, q, kTableChunk});
                  ul->item_cost_table.push_back((double)u.n_m);
                }
                ul->item_cost_table.back() +=
                    (double)nq * 12.0 * (E + 2) * (double)u.n_m / (double)L +
                    (double)u.n_targets * nq * 64.0;
              } else {
                // one item per `chunk` tiles: one library staging (when it
                // fits a shared-memory tile), then per tile the search and the
                // per-target epilogue
                if (q % chunk == 0) {
                  ul->items.push_back(WorkItem{uidx, q, chunk});
                  ul->item_cost.push_back(64.0 * E * (double)L);
                }
                ul->item_cost.back() += (double)L * (double)nq * (2.0 * E + 1.0) +
                                        (double)u.n_targets * nq * 64.0;
              }
            }
            if (u.table_R == 0) {
              ul->brute_flops += 3.0 * E * (double)u.n_m * (double)L;
              ul->brute_pairs += (double)u.n_m * (double)L;
            } else {
              ul->table_queries += u.n_m;
            }
            ul->search_queries += u.n_m;
            if (u.table_R == 0) ul->lib_total += L;
            ul->part_total += (int64_t)u.n_tiles * u.n_targets;
            ul->emin = std::min(ul->emin, E);
            ul->emax = std::max(ul->emax, E);
            ul->max_nm = std::max(ul->max_nm, u.n_m);
            ul->pairs += (double)u.n_m * (double)L;
            ul->flops += 3.0 * E * (double)u.n_m * (double)L;
            ul->units.push_back(u);
          }
        }
        if (!grouped) continue;
        // Scan groups: consecutive units of this (j, E, tau) that read the table,
        // whatever their L (the lanes of a partly filled group would idle; the
        // walk of a mixed one is as long as its smallest L's).
        // Tiles per item: one copy of the membership words (about 4 % of a tile's
        // time) against the balance of eight items per CTA slot.
        const int64_t slots = scan_tiles[E] / (8 * 2 * kSms);
        const int32_t chunk =
            tp.size() > 1 ? 1 : (int32_t)std::min<int64_t>(std::max<int64_t>(slots, 1), kScanChunk);
        const size_t group = tp.size() > 1 ? (size_t)lanes_group : (size_t)kScanGroup;
        for (size_t a = first_unit; a < ul->units.size();) {
          if (ul->units[a].table_R == 0) {
            ++a;
            continue;
          }
          size_t b = a;
          int32_t lmin = ul->units[a].L;
          for (; b < ul->units.size() && b - a < group && ul->units[b].table_R > 0; ++b) {
            ul->units[b].words_off = ul->words_total;
            lmin = std::min(lmin, ul->units[b].L);
          }
          const UnitDesc& u = ul->units[a];
          ul->words_total += member_words(u.n_m);
          ul->member_groups.push_back(MemberGroup{(int32_t)a, (int32_t)(b - a)});
          for (int32_t q = 0; q < u.n_tiles; q += chunk) {
            ul->items_table.push_back(
                WorkItem{(int32_t)a, q, (int32_t)(b - a) | (tp.size() > 1 ? 0 : chunk << 8)});
            ul->item_cost_table.push_back(std::min(chunk, u.n_tiles - q) *
                                          (64.0 + (E + 4.0) * u.n_m / lmin +
                                           (tp.size() > 1 ? 1.5 * (double)(b - a) * u.n_targets : 0.0)));
          }
          a = b;
        }
      }
  }
}

void sort_items(UnitList* ul) {
  for (UnitDesc& u : ul->units)
    if (u.table_R > 0) u.lib_off = ul->lib_total;  // one slot behind the lists
  std::stable_sort(ul->tables.begin(), ul->tables.end(), [](const TableJob& a, const TableJob& b) {
    const int ra = UnitList::table_rcap(a.R), rb = UnitList::table_rcap(b.R);
    if (ra != rb) return ra < rb;
    if (a.E != b.E) return a.E < b.E;
    return a.R < b.R;
  });
  // Brute-force items: grouped by E (one single-E kernel launch per group,
  // in the stream's order), larger items first within a group.
  {
    std::vector<int64_t> order(ul->items.size());
    for (size_t q = 0; q < order.size(); ++q) order[q] = (int64_t)q;
    std::stable_sort(order.begin(), order.end(), [&](int64_t a, int64_t b) {
      const int32_t ea = ul->units[(size_t)ul->items[(size_t)a].unit].E;
      const int32_t eb = ul->units[(size_t)ul->items[(size_t)b].unit].E;
      if (ea != eb) return ea > eb;
      const Targets ta = ul->targets_of(ul->items[(size_t)a]);
      const Targets tb = ul->targets_of(ul->items[(size_t)b]);
      if (ta != tb) return ta > tb;
      return ul->item_cost[(size_t)a] > ul->item_cost[(size_t)b];
    });
    std::vector<WorkItem> sorted(order.size());
    std::vector<double> cost(order.size());
    for (size_t q = 0; q < order.size(); ++q) {
      sorted[q] = ul->items[(size_t)order[q]];
      cost[q] = ul->item_cost[(size_t)order[q]];
    }
    ul->items.swap(sorted);
    ul->item_cost.swap(cost);
    ul->groups = ul->group_items(ul->items);
  }
  // Table items: grouped by E (one launch per E and kind), then by table and,
  // for the scan, by query tiles, so that all realizations that walk a row do
  // so while it is in L2; larger items first.
  std::vector<int64_t> order(ul->items_table.size());
  for (size_t q = 0; q < order.size(); ++q) order[q] = (int64_t)q;
  std::stable_sort(order.begin(), order.end(), [&](int64_t a, int64_t b) {
    const UnitDesc& ua = ul->units[(size_t)ul->items_table[(size_t)a].unit];
    const UnitDesc& ub = ul->units[(size_t)ul->items_table[(size_t)b].unit];
    if (ua.E != ub.E) return ua.E > ub.E;
    const WorkItem &wa = ul->items_table[(size_t)a], &wb = ul->items_table[(size_t)b];
    const Targets ta = ul->targets_of(wa), tb = ul->targets_of(wb);
    if (ta != tb) return ta > tb;
    if (ua.table_off != ub.table_off) return ua.table_off < ub.table_off;
    if ((ta == Targets::kOne || ta == Targets::kGrouped) && wa.tile != wb.tile) return wa.tile < wb.tile;
    return ul->item_cost_table[(size_t)a] > ul->item_cost_table[(size_t)b];
  });
  std::vector<WorkItem> sorted(order.size());
  for (size_t q = 0; q < order.size(); ++q) sorted[q] = ul->items_table[(size_t)order[q]];
  ul->items_table.swap(sorted);
  ul->groups_table = ul->group_items(ul->items_table);
}

// Search launches of one run, at most: per E, brute force of few or many
// targets, tables of one, few or many, or of many in groups.
constexpr int kMaxSearchLaunches = 6 * kMaxE;

// Device arena layout for a unit list.
struct Arena {
  size_t series = 0, units = 0, items = 0, lib = 0, part = 0, rho = 0, err = 0,
         counter = 0, scratch = 0, order = 0, orders = 0, targets = 0, table = 0, tables = 0,
         items_table = 0, order_scratch = 0, obs = 0, obs_stat = 0, obs_jobs = 0, series_jobs = 0,
         scales = 0, st = 0, table_dist = 0, stats = 0, inverse = 0, bits = 0, words = 0,
         member_groups = 0, points = 0,
         total = 0;
};

Arena layout(int64_t series_elems, const UnitList& ul, int64_t n_rho, int64_t scratch_floats) {
  Arena a;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o = align_up(o + bytes, 256);
    return at;
  };
  a.series = take(sizeof(float) * (size_t)series_elems);
  a.units = take(sizeof(UnitDesc) * ul.units.size());
  a.items = take(sizeof(WorkItem) * ul.items.size());
  a.lib = take(sizeof(int32_t) * (size_t)(ul.lib_total + ul.lib_scratch));
  a.bits = take(sizeof(uint32_t) * (size_t)ul.bits_total);
  a.words = take(sizeof(uint32_t) * (size_t)ul.words_total);
  a.member_groups = take(sizeof(MemberGroup) * ul.member_groups.size());
  a.part = take(2 * sizeof(float4) * (size_t)ul.part_total);
  a.rho = take(sizeof(double) * (size_t)n_rho);
  a.err = take(sizeof(int32_t));
  a.counter = take(kMaxSearchLaunches * sizeof(uint32_t));
  a.scratch = take(sizeof(float) * (size_t)scratch_floats);
  a.order = take(sizeof(int32_t) * (size_t)ul.order_total);
  a.inverse = take(ul.tables.empty() ? 0 : sizeof(int32_t) * (size_t)ul.order_total);
  a.order_scratch = take(sizeof(unsigned long long) * (size_t)ul.order_scratch_total);
  a.orders = take(sizeof(OrderJob) * ul.orders.size());
  a.targets = take(sizeof(TargetDesc) * ul.targets.size());
  a.table = take(ul.table_elem() * (size_t)ul.table_total);
  a.table_dist = take((ul.table_tv ? sizeof(float2) : sizeof(float)) * (size_t)ul.table_total);
  a.points = take(sizeof(float) * (size_t)ul.points_total);
  a.tables = take(sizeof(TableJob) * ul.tables.size());
  a.items_table = take(sizeof(WorkItem) * ul.items_table.size());
  a.obs = take(sizeof(float2) * (size_t)knn_block_threads() * (size_t)ul.obs_total);
  a.obs_stat = take(sizeof(ObsStat) * (size_t)ul.obs_total);
  a.obs_jobs = take(sizeof(ObsJob) * ul.obs_jobs.size());
  a.series_jobs = take(sizeof(SeriesJob) * ul.series_jobs.size());
  a.scales = take(sizeof(SeriesScale) * ul.series_jobs.size());
  a.st = take(sizeof(float) * (size_t)ul.st_total);
  a.stats = take(sizeof(unsigned long long) * kStatCount);
  a.total = o;
  return a;
}

}  // namespace

namespace ccm {
void set_last_error(const char* msg) { t_err = msg; }
}  // namespace ccm

// Per-E kernel parameters chosen by the autotuner (results do not depend on them).
struct Tuning {
  int32_t variant[kMaxE + 1];
  int32_t merge_at[kMaxE + 1];
  bool known[kMaxE + 1];  // chosen by measurement (here or from the cache)
};

Tuning default_tuning() {
  Tuning t;
  for (int e = 0; e <= kMaxE; ++e) {
    t.variant[e] = kDefaultVariant;
    t.merge_at[e] = kDefaultMergeAt;
    t.known[e] = false;
  }
  return t;
}

// ================================================================ context ===
struct Job;
struct Batch;

struct ccm_context {
  int device = 0;
  std::string device_name;
  Tuning tuning = default_tuning();  // per-E choices known to this context (cache + runs)
  size_t budget = 0;
  size_t used = 0;
  int sm_count = 0;
  std::mutex mu;  // budget, job table, queue, batches
  std::condition_variable cv;
  // serving state
  std::thread server;
  bool server_started = false;
  bool stop = false;
  uint64_t next_ticket = 1;
  std::map<uint64_t, std::shared_ptr<Job>> jobs;
  std::deque<std::shared_ptr<Job>> queue;
  std::list<std::shared_ptr<Batch>> inflight;
  std::vector<cudaStream_t> streams;       // low priority: batches of large jobs
  std::vector<cudaStream_t> fast_streams;  // high priority: batches of small jobs
  size_t next_stream = 0, next_fast = 0;
  int max_inflight = 8;
  double batch_pairs = 5.0e10;             // query-library pairs per batch of small jobs
  // Test hook (CCM_FAULT_INJECT_BATCH, read at creation): the launch of batch
  // number inject_batch (0-based, in launch order) fails on the host as if a
  // CUDA call had returned an error; -1: off.  No device work is faulted.
  int64_t inject_batch = -1;
  int64_t batches_launched = 0;
  // Pinned staging buffers are pooled: cudaMallocHost/cudaFreeHost may
  // synchronise the device, which would stall polls and new batches behind a
  // running large job.  Size classes are powers of two.
  std::mutex pool_mu;
  std::multimap<size_t, void*> pool_free;
  std::vector<void*> pool_all;
};

namespace {
// What a plan (or served job) may hold beside what it needs: tables of a quarter of
// the context's budget and the time-major copy of its series; where the plan does
// not fit, smaller tables, then none, then no copy either.
constexpr int kRooms = 4;
Room room_of(const ccm_context* ctx, int attempt) {
  constexpr double kTables[kRooms] = {0.25, 0.025, 0.0, 0.0};
  return Room{kTables[attempt] * (double)ctx->budget, attempt < 3};
}
// No attempt after this one gives a smaller plan.
bool barest(const UnitList& ul) { return ul.tables.empty() && ul.st_total == 0; }
}  // namespace

namespace {

size_t pool_class(size_t bytes) {
  size_t c = 256;
  while (c < bytes) c <<= 1;
  return c;
}

void* pinned_get(ccm_context* ctx, size_t bytes) {
  const size_t c = pool_class(bytes);
  std::lock_guard<std::mutex> g(ctx->pool_mu);
  auto it = ctx->pool_free.find(c);
  if (it != ctx->pool_free.end()) {
    void* ptr = it->second;
    ctx->pool_free.erase(it);
    return ptr;
  }
  void* ptr = nullptr;
  if (cudaMallocHost(&ptr, c) != cudaSuccess) return nullptr;
  ctx->pool_all.push_back(ptr);
  return ptr;
}

void pinned_put(ccm_context* ctx, void* ptr, size_t bytes) {
  if (!ptr) return;
  std::lock_guard<std::mutex> g(ctx->pool_mu);
  ctx->pool_free.emplace(pool_class(bytes), ptr);
}

ccm_status reserve(ccm_context* ctx, size_t bytes) {
  std::lock_guard<std::mutex> g(ctx->mu);
  if (bytes > ctx->budget)
    return fail(CCM_ETOOLARGE, "footprint " + std::to_string(bytes) + " B exceeds budget " +
                                   std::to_string(ctx->budget) + " B");
  if (ctx->used + bytes > ctx->budget)
    return fail(CCM_ENOMEM, "budget in use: " + std::to_string(ctx->used) + " of " +
                                std::to_string(ctx->budget) + " B");
  ctx->used += bytes;
  return CCM_OK;
}

void release(ccm_context* ctx, size_t bytes) {
  std::lock_guard<std::mutex> g(ctx->mu);
  ctx->used -= std::min(ctx->used, bytes);
}

}  // namespace

// =================================================================== plan ===
struct ccm_plan_s {
  ccm_context* ctx = nullptr;
  ProblemCopy pc;
  UnitList ul;
  Arena ar;
  char* d_arena = nullptr;
  cudaStream_t stream = nullptr;
  cudaGraphExec_t graph = nullptr;
  cudaEvent_t ev[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};  // stage boundaries
  int grid = 0, grid_table = 0, grid_scan = 0;
  Tuning tuning = default_tuning();
  bool tuned = false;
  std::mutex run_mu;
  ccm_plan_info info{};
};

namespace {

SamplerParams sampler_params(char* base, const Arena& ar, const UnitList& ul) {
  SamplerParams sp{};
  sp.window = ul.sampler_window;
  sp.units = reinterpret_cast<const UnitDesc*>(base + ar.units);
  sp.targets = reinterpret_cast<const TargetDesc*>(base + ar.targets);
  sp.order = reinterpret_cast<const int32_t*>(base + ar.order);
  sp.lib = reinterpret_cast<int32_t*>(base + ar.lib);
  sp.bits = reinterpret_cast<uint32_t*>(base + ar.bits);
  sp.err = reinterpret_cast<int32_t*>(base + ar.err);
  return sp;
}

KnnParams knn_params(char* base, const Arena& ar, const UnitList& ul, int persistent,
                     const Tuning& tn) {
  KnnParams kp{};
  kp.series = reinterpret_cast<const float*>(base + ar.series);
  kp.units = reinterpret_cast<const UnitDesc*>(base + ar.units);
  kp.targets = reinterpret_cast<const TargetDesc*>(base + ar.targets);
  kp.items = reinterpret_cast<const WorkItem*>(base + ar.items);
  kp.n_items = (int64_t)ul.items.size();
  kp.lib = reinterpret_cast<const int32_t*>(base + ar.lib);
  kp.order = reinterpret_cast<const int32_t*>(base + ar.order);
  kp.bits = reinterpret_cast<const uint32_t*>(base + ar.bits);
  kp.words = reinterpret_cast<const uint32_t*>(base + ar.words);
  kp.window = ul.window ? 1 : 0;
  kp.table = base + ar.table;
  kp.table_dist = reinterpret_cast<const float*>(base + ar.table_dist);
  kp.table_pairs = ul.table_tv ? 1 : 0;
  kp.table_u16 = ul.table_u16();
  kp.partials = reinterpret_cast<float4*>(base + ar.part);
  kp.obs = reinterpret_cast<const float2*>(base + ar.obs);
  kp.obs_stat = reinterpret_cast<const ObsStat*>(base + ar.obs_stat);
  kp.st = reinterpret_cast<const float*>(base + ar.st);
  kp.item_counter = reinterpret_cast<uint32_t*>(base + ar.counter);
  kp.err = reinterpret_cast<int32_t*>(base + ar.err);
  kp.persistent = persistent;
  kp.prune = 1;
  for (int e = 0; e <= kMaxE; ++e) {
    kp.merge_at[e] = tn.merge_at[e];
    kp.variant[e] = tn.variant[e];
  }
  return kp;
}

// Query order and target series, then the observed-value records.
cudaError_t enqueue_order(char* base, const Arena& ar, const UnitList& ul, LaunchStream s) {
  SeriesScale* scales = reinterpret_cast<SeriesScale*>(base + ar.scales);
  const cudaError_t e =
      launch_order(reinterpret_cast<const float*>(base + ar.series),
                   reinterpret_cast<const OrderJob*>(base + ar.orders), (int64_t)ul.orders.size(),
                   ul.max_nm, reinterpret_cast<int32_t*>(base + ar.order),
                   ul.tables.empty() ? nullptr : reinterpret_cast<int32_t*>(base + ar.inverse),
                   reinterpret_cast<unsigned long long*>(base + ar.order_scratch),
                   reinterpret_cast<const SeriesJob*>(base + ar.series_jobs),
                   (int64_t)ul.series_jobs.size(), scales, reinterpret_cast<float*>(base + ar.st), s);
  if (e != cudaSuccess) return e;
  return launch_obs(reinterpret_cast<const float*>(base + ar.series),
                    reinterpret_cast<const int32_t*>(base + ar.order),
                    reinterpret_cast<const ObsJob*>(base + ar.obs_jobs),
                    (int64_t)ul.obs_jobs.size(), ul.obs_total, scales,
                    reinterpret_cast<float2*>(base + ar.obs),
                    reinterpret_cast<ObsStat*>(base + ar.obs_stat), s);
}

// A second branch of a captured run: the tables need only the query orders, so
// they are built beside the sampler and the brute-force searches.  Short
// manifolds leave part of the chip idle in each of these (N = 1000 0.171 ->
// 0.159 ms a run, N = 2347 0.635 -> 0.570, 64 variables of N = 5000 55.5 -> 53.5);
// long ones do not (N = 10^4 161.6 and 161.6, N = 10^5 87.6 -> 89.1) and keep one
// stream.
constexpr int kBranchMaxNm = 8192;
struct TableBranch {
  cudaStream_t s = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
  cudaError_t create() {
    cudaError_t e = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&join, cudaEventDisableTiming);
    return e;
  }
  ~TableBranch() {
    if (join) cudaEventDestroy(join);
    if (fork) cudaEventDestroy(fork);
    if (s) cudaStreamDestroy(s);
  }
};

// Enqueue sampler + fused kernel for a whole unit list on stream s.
// Stage events (optional): ev[0] start, ev[5] after order, observed moments and
// table build, ev[1] before the sampler, ev[2] after it, ev[3] after the
// brute-force launch, ev[4] after the table-scan launch.
ccm_status enqueue_sweep(char* base, const Arena& ar, const UnitList& ul, const Tuning& tn,
                         int grid, int grid_table, int grid_scan, int persistent, int32_t* dbg_lib,
                         int32_t* dbg_nbr, float* dbg_xhat, cudaStream_t s,
                         cudaEvent_t* ev = nullptr, bool capturing = false,
                         bool stats = false, const TableBranch* branch = nullptr) {
  const LaunchStream ls(s, persistent && !capturing);
  // the table builds: on the stream itself, or beside sampler and brute force
  const LaunchStream ts = branch ? LaunchStream(branch->s) : ls;
  // Inside stream capture an event record becomes a graph node only with the
  // external flag; outside capture the plain record is the valid form.
  auto record = [&](cudaEvent_t e, cudaStream_t on) {
    return capturing ? cudaEventRecordWithFlags(e, on, cudaEventRecordExternal)
                     : cudaEventRecord(e, on);
  };
  CCM_CUDA(cudaMemsetAsync(base + ar.err, 0, sizeof(int32_t), s));
  CCM_CUDA(cudaMemsetAsync(base + ar.counter, 0, kMaxSearchLaunches * sizeof(uint32_t), s));
  if (stats) CCM_CUDA(cudaMemsetAsync(base + ar.stats, 0, sizeof(unsigned long long) * kStatCount, s));
  if (ev) CCM_CUDA(record(ev[0], s));
  CCM_CUDA(enqueue_order(base, ar, ul, ls));
  if (branch) {
    CCM_CUDA(cudaEventRecord(branch->fork, s));
    CCM_CUDA(cudaStreamWaitEvent(branch->s, branch->fork, 0));
  }
  if (!ul.tables.empty())
    CCM_CUDA(launch_table_points(reinterpret_cast<const float*>(base + ar.series),
                                 reinterpret_cast<const TableJob*>(base + ar.tables),
                                 (int64_t)ul.tables.size(), ul.table_max_nm,
                                 reinterpret_cast<const int32_t*>(base + ar.order),
                                 reinterpret_cast<float*>(base + ar.points), ts));
  for (size_t g0 = 0; g0 < ul.tables.size();) {  // one launch per (size class, E)
    const int rc = UnitList::table_rcap(ul.tables[g0].R), te = ul.tables[g0].E;
    size_t g1 = g0;
    int nm = 0, rmax = 0;
    int64_t rows = 0;
    for (; g1 < ul.tables.size() && UnitList::table_rcap(ul.tables[g1].R) == rc &&
           ul.tables[g1].E == te && g1 - g0 < 65535;
         ++g1) {
      nm = std::max(nm, ul.tables[g1].n_m);
      rmax = std::max(rmax, ul.tables[g1].R);
      rows += ul.tables[g1].n_m;
    }
    CCM_CUDA(launch_table_build(reinterpret_cast<const float*>(base + ar.series),
                                reinterpret_cast<const TableJob*>(base + ar.tables) + g0,
                                (int64_t)(g1 - g0), rows, te, nm, rmax,
                                reinterpret_cast<const float*>(base + ar.points),
                                reinterpret_cast<const int32_t*>(base + ar.order),
                                reinterpret_cast<const int32_t*>(base + ar.inverse),
                                base + ar.table, reinterpret_cast<float*>(base + ar.table_dist),
                                ul.table_tv ? 1 : 0, ul.table_u16(),
                                reinterpret_cast<int32_t*>(base + ar.err), ts));
    g0 = g1;
  }
  if (ev) CCM_CUDA(record(ev[5], ts.s));
  if (branch) CCM_CUDA(cudaEventRecord(branch->join, branch->s));
  if (ev) CCM_CUDA(record(ev[1], s));
  SamplerParams sp = sampler_params(base, ar, ul);
  sp.dbg_lib = dbg_lib;
  CCM_CUDA(launch_sampler(sp, 0, (int64_t)ul.units.size(), ul.max_nm, ls));
  if (!ul.member_groups.empty())
    CCM_CUDA(launch_member_words(reinterpret_cast<const UnitDesc*>(base + ar.units),
                                 reinterpret_cast<const MemberGroup*>(base + ar.member_groups),
                                 (int64_t)ul.member_groups.size(), ul.table_max_nm, sp.bits,
                                 reinterpret_cast<uint32_t*>(base + ar.words), ls));
  if (ev) CCM_CUDA(record(ev[2], s));
  KnnParams kp = knn_params(base, ar, ul, persistent, tn);
  kp.dbg_nbr = dbg_nbr;
  kp.dbg_xhat = dbg_xhat;
  if (stats) kp.stats = reinterpret_cast<unsigned long long*>(base + ar.stats);
  // One launch per E (a kernel specialised for one E keeps its registers for
  // that E); each drains its own queue, larger items first, so the launches
  // follow each other with short tails.
  uint32_t* counter = reinterpret_cast<uint32_t*>(base + ar.counter);  // one per launch
  for (const ItemGroup& ig : ul.groups) {
    KnnParams ke = kp;
    ke.items = kp.items + ig.first;
    ke.n_items = ig.count;
    ke.item_counter = counter++;
    const int g = persistent ? grid : (int)std::min<int64_t>(ig.count, 0x7fffffff);
    CCM_CUDA(launch_knn(ke, ig.E, ig.targets == Targets::kMany, g, ls));
  }
  if (ev) CCM_CUDA(record(ev[3], s));
  if (branch) CCM_CUDA(cudaStreamWaitEvent(s, branch->join, 0));
  for (const ItemGroup& ig : ul.groups_table) {
    KnnParams kt = kp;
    kt.items = reinterpret_cast<const WorkItem*>(base + ar.items_table) + ig.first;
    kt.n_items = ig.count;
    kt.item_counter = counter++;
    const int g = persistent ? grid_table : (int)std::min<int64_t>(ig.count, 0x7fffffff);
    if (ig.targets == Targets::kOne)
      CCM_CUDA(launch_knn_scan(kt, ig.E, ig.max_nm, persistent ? grid_scan : g, ls));
    else if (ig.targets == Targets::kGrouped)
      CCM_CUDA(launch_knn_group(kt, ig.E, ig.max_nm, persistent ? grid_scan / 2 : g, ls));
    else
      CCM_CUDA(launch_knn_table(kt, ig.E, ig.max_nm, ig.targets == Targets::kMany, g, ls));
  }
  CCM_CUDA(launch_rho(kp.units, kp.targets, (int64_t)ul.targets.size(), (ul.max_nm + 255) / 256, kp.partials,
                      kp.obs_stat,
                      reinterpret_cast<double*>(base + ar.rho), ls));
  if (ev) CCM_CUDA(record(ev[4], s));
  return CCM_OK;
}

ccm_status check_err_flag(char* base, const Arena& ar, cudaStream_t s) {
  int32_t err = 0;
  CCM_CUDA(cudaMemcpyAsync(&err, base + ar.err, sizeof(err), cudaMemcpyDeviceToHost, s));
  CCM_CUDA(cudaStreamSynchronize(s));
  if (err != 0) return fail(CCM_ECUDA, "kernel reported error flag " + std::to_string(err));
  return CCM_OK;
}

int persistent_grid(ccm_context* ctx, int emin, int emax) {
  int per_sm = 1 << 30;  // the smallest occupancy of the plan's kernels
  for (int E = std::max(emin, 1); E <= std::min(emax, kMaxE); ++E) {
    int c = 1;
    if (knn_occupancy(E, &c) != cudaSuccess || c < 1) c = 1;
    per_sm = std::min(per_sm, c);
  }
  if (per_sm == (1 << 30)) per_sm = 1;
  return ctx->sm_count * per_sm;
}

}  // namespace

// ============================================================== autotuner ===
namespace {

// Per E the tuner times the kernel variants (narrow / wide) and merge triggers
// on a stratified sample of the plan's own work items and keeps the fastest.
// Every candidate computes the same result; only the time differs.  Choices
// are cached per (device name, kernel revision, E) in a tab-separated file:
// $CCM_AUTOTUNE_CACHE, else ~/.cache/ccm_gb300/autotune.tsv.  The revision (a hash
// of the search kernels' sources, from build.py) keeps the choices measured with
// other kernels from being taken for these.
#ifndef CCM_KERNEL_REVISION
#define CCM_KERNEL_REVISION "unknown"
#endif
constexpr char kRevision[] = "r" CCM_KERNEL_REVISION;
std::string cache_path() {
  if (const char* p = getenv("CCM_AUTOTUNE_CACHE")) return p;
  const char* home = getenv("HOME");
  return std::string(home ? home : "/tmp") + "/.cache/ccm_gb300/autotune.tsv";
}

void load_cache(ccm_context* ctx) {
  FILE* f = fopen(cache_path().c_str(), "r");
  if (!f) return;
  char line[512];
  while (fgets(line, sizeof(line), f)) {
    char name[256], revision[64];
    int E = 0, v = 0, ma = 0;
    if (sscanf(line, "%255[^\t]\t%63[^\t]\t%d\t%d\t%d", name, revision, &E, &v, &ma) == 5 &&
        ctx->device_name == name && std::strcmp(revision, kRevision) == 0 && E >= 1 && E <= kMaxE && v >= 0 && v <= 1 && ma >= 1 &&
        ma <= 16) {
      ctx->tuning.variant[E] = v;
      ctx->tuning.merge_at[E] = ma;
      ctx->tuning.known[E] = true;
    }
  }
  fclose(f);
}

void save_cache(const ccm_context* ctx, int E, int v, int ma) {
  const std::string path = cache_path();
  const size_t slash = path.rfind('/');
  if (slash != std::string::npos) {  // mkdir -p of the parent, best effort
    std::string dir = path.substr(0, slash);
    for (size_t q = 1; q <= dir.size(); ++q)
      if (q == dir.size() || dir[q] == '/') {
        const std::string d = dir.substr(0, q);
        (void)mkdir(d.c_str(), 0755);
      }
  }
  FILE* f = fopen(path.c_str(), "a");
  if (!f) return;
  fprintf(f, "%s\t%s\t%d\t%d\t%d\n", ctx->device_name.c_str(), kRevision, E, v, ma);
  fclose(f);
}

constexpr double kTunePairs = 2.0e11;   // plans smaller than this use known or default choices

// The brute-force items of one E that the tuner samples from: of one kind (of many
// targets only where a plan has no others of this E).
std::vector<WorkItem> tuning_items(const UnitList& ul, int E, Targets* kind) {
  *kind = Targets::kMany;
  for (const ItemGroup& ig : ul.groups)
    if (ig.E == E) *kind = std::min(*kind, ig.targets);
  std::vector<WorkItem> all;
  for (const ItemGroup& ig : ul.groups)
    if (ig.E == E && ig.targets == *kind)
      all.insert(all.end(), ul.items.begin() + ig.first, ul.items.begin() + ig.first + ig.count);
  return all;
}

ccm_status autotune(ccm_plan_s* pl, cudaStream_t s) {
  ccm_context* ctx = pl->ctx;
  char* base = pl->d_arena;
  const Arena& ar = pl->ar;
  const UnitList& ul = pl->ul;
  const int want = 6 * ctx->sm_count;
  // an E whose libraries all read tables has nothing to measure
  bool any = false;
  for (int E = ul.emin; E <= ul.emax; ++E) {
    Targets kind;
    any |= !pl->tuning.known[E] && (int)tuning_items(ul, E, &kind).size() >= want;
  }
  if (!any) return CCM_OK;
  // libraries and query orders for the timing launches
  CCM_CUDA(enqueue_order(base, ar, ul, s));
  SamplerParams sp = sampler_params(base, ar, ul);
  CCM_CUDA(launch_sampler(sp, 0, (int64_t)ul.units.size(), ul.max_nm, s));
  WorkItem* d_items = nullptr;
  CCM_CUDA(cudaMallocAsync(&d_items, sizeof(WorkItem) * (size_t)want, s));
  cudaEvent_t e0, e1;
  CCM_CUDA(cudaEventCreate(&e0));
  CCM_CUDA(cudaEventCreate(&e1));
  ccm_status st = CCM_OK;
  for (int E = ul.emin; E <= ul.emax && st == CCM_OK; ++E) {
    if (pl->tuning.known[E]) continue;
    Targets kind;
    const std::vector<WorkItem> all = tuning_items(ul, E, &kind);
    if ((int)all.size() < want) continue;
    std::vector<WorkItem> sample;  // evenly spaced over the cost-sorted list
    for (int q = 0; q < want; ++q) sample.push_back(all[(size_t)q * all.size() / (size_t)want]);
    cudaError_t ce = cudaMemcpyAsync(d_items, sample.data(), sizeof(WorkItem) * sample.size(),
                                     cudaMemcpyHostToDevice, s);
    if (ce != cudaSuccess) { st = fail(CCM_ECUDA, cudaGetErrorString(ce)); break; }
    float best = 1e30f;
    int best_v = pl->tuning.variant[E], best_ma = pl->tuning.merge_at[E];
    for (int v = 0; v < 2; ++v)
      for (int ma : {1, 2, 4, 8}) {
        Tuning tn = pl->tuning;
        tn.variant[E] = v;
        tn.merge_at[E] = ma;
        KnnParams kp = knn_params(base, ar, ul, 0, tn);
        kp.items = d_items;
        kp.n_items = (int64_t)sample.size();
        float ms = 0.f;
        for (int rep = 0; rep < 2 && ce == cudaSuccess; ++rep) {  // warm-up, then timed
          ce = cudaEventRecord(e0, s);
          if (ce == cudaSuccess) ce = launch_knn(kp, E, kind == Targets::kMany, (int)sample.size(), s);
          if (ce == cudaSuccess) ce = cudaEventRecord(e1, s);
          if (ce == cudaSuccess) ce = cudaEventSynchronize(e1);
          if (ce == cudaSuccess) ce = cudaEventElapsedTime(&ms, e0, e1);
        }
        if (ce != cudaSuccess) break;
        if (ms < best) {
          best = ms;
          best_v = v;
          best_ma = ma;
        }
      }
    if (ce != cudaSuccess) { st = fail(CCM_ECUDA, cudaGetErrorString(ce)); break; }
    pl->tuning.variant[E] = best_v;
    pl->tuning.merge_at[E] = best_ma;
    pl->tuning.known[E] = true;
    {
      std::lock_guard<std::mutex> g(ctx->mu);
      ctx->tuning.variant[E] = best_v;
      ctx->tuning.merge_at[E] = best_ma;
      ctx->tuning.known[E] = true;
    }
    save_cache(ctx, E, best_v, best_ma);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFreeAsync(d_items, s);
  if (st == CCM_OK) CCM_CUDA(cudaStreamSynchronize(s));
  return st;
}

}  // namespace

// ==================================================================== ABI ===
extern "C" {

const char* ccm_last_error(void) { return t_err.c_str(); }

const char* ccm_version(void) { return "ccm-gb300 0.1 (sm_103a)"; }

ccm_status ccm_context_create(int device, size_t hbm_budget_bytes, ccm_context** out) {
  if (!out) return fail(CCM_EINVAL, "out is NULL");
  *out = nullptr;
  int count = 0;
  CCM_CUDA(cudaGetDeviceCount(&count));
  if (device < 0 || device >= count) return fail(CCM_EINVAL, "no such device");
  CCM_CUDA(cudaSetDevice(device));
  cudaDeviceProp prop;
  CCM_CUDA(cudaGetDeviceProperties(&prop, device));
  if (prop.major < 10) return fail(CCM_EINVAL, "needs a Blackwell (sm_10x) GPU");
  CCM_CUDA(sampler_prepare());
  CCM_CUDA(knn_prepare());
  CCM_CUDA(order_prepare());
  CCM_CUDA(table_prepare());
  CCM_CUDA(convergence_prepare());
  CCM_CUDA(knn_table_prepare());
  CCM_CUDA(knn_scan_prepare());
  CCM_CUDA(knn_group_prepare());
  size_t free_b = 0, total_b = 0;
  CCM_CUDA(cudaMemGetInfo(&free_b, &total_b));
  std::unique_ptr<ccm_context> ctx(new ccm_context());
  ctx->device = device;
  ctx->device_name = prop.name;
  ctx->sm_count = prop.multiProcessorCount;
  load_cache(ctx.get());
  if (const char* env = getenv("CCM_FAULT_INJECT_BATCH")) ctx->inject_batch = atoll(env);
  ctx->budget = hbm_budget_bytes ? hbm_budget_bytes : (size_t)(0.9 * (double)free_b);
  *out = ctx.release();
  return CCM_OK;
}

ccm_status ccm_plan(ccm_context* ctx, const ccm_problem* prob, ccm_plan_t** out) {
  if (!ctx || !out) return fail(CCM_EINVAL, "NULL argument");
  *out = nullptr;
  std::unique_ptr<ccm_plan_s> pl(new ccm_plan_s());
  pl->ctx = ctx;
  ccm_status st = copy_problem(prob, &pl->pc);
  if (st != CCM_OK) return st;
  const int64_t series_elems = (int64_t)pl->pc.V * pl->pc.n;
  CCM_CUDA(cudaSetDevice(ctx->device));
  // where the plan does not fit, once more with less room (room_of)
  cudaError_t e = cudaSuccess;
  for (int attempt = 0; attempt < kRooms; ++attempt) {
    pl->ul = UnitList();
    append_units(pl->pc, 0, 0, &pl->ul, room_of(ctx, attempt));
    sort_items(&pl->ul);
    pl->ar = layout(series_elems, pl->ul, pl->ul.n_rho, pl->ul.max_nm);
    const bool last = barest(pl->ul);
    st = reserve(ctx, pl->ar.total);
    if (st != CCM_OK) {
      if (last) return st;
      continue;
    }
    e = cudaMalloc(&pl->d_arena, pl->ar.total);
    if (e == cudaSuccess) break;
    pl->d_arena = nullptr;
    release(ctx, pl->ar.total);
    if (last) return fail(CCM_ENOMEM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
    (void)cudaGetLastError();  // reported by the next attempt if it fails too
  }
  e = cudaStreamCreateWithFlags(&pl->stream, cudaStreamNonBlocking);
  for (int q = 0; q < 6 && e == cudaSuccess; ++q) e = cudaEventCreate(&pl->ev[q]);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.units, pl->ul.units.data(),
                   sizeof(UnitDesc) * pl->ul.units.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.items, pl->ul.items.data(),
                   sizeof(WorkItem) * pl->ul.items.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.orders, pl->ul.orders.data(),
                   sizeof(OrderJob) * pl->ul.orders.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.targets, pl->ul.targets.data(),
                   sizeof(TargetDesc) * pl->ul.targets.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.tables, pl->ul.tables.data(),
                   sizeof(TableJob) * pl->ul.tables.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.obs_jobs, pl->ul.obs_jobs.data(),
                   sizeof(ObsJob) * pl->ul.obs_jobs.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.items_table, pl->ul.items_table.data(),
                   sizeof(WorkItem) * pl->ul.items_table.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.member_groups, pl->ul.member_groups.data(),
                   sizeof(MemberGroup) * pl->ul.member_groups.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(pl->d_arena + pl->ar.series_jobs, pl->ul.series_jobs.data(),
                   sizeof(SeriesJob) * pl->ul.series_jobs.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cudaFree(pl->d_arena);
    if (pl->stream) cudaStreamDestroy(pl->stream);
    release(ctx, pl->ar.total);
    return fail(CCM_ECUDA, std::string("plan set-up: ") + cudaGetErrorString(e));
  }
  pl->grid = persistent_grid(ctx, pl->ul.emin, pl->ul.emax);
  {
    int per_sm = 1;
    if (knn_table_occupancy(pl->ul.table_max_nm, pl->ul.lane_targets, &per_sm) != cudaSuccess || per_sm < 1)
      per_sm = 1;
    pl->grid_table = ctx->sm_count * per_sm;
    pl->grid_scan = ctx->sm_count * 2;
  }
  {
    std::lock_guard<std::mutex> g(ctx->mu);
    pl->tuning = ctx->tuning;
  }
  ccm_plan_info& in = pl->info;
  in.n_units = pl->ul.n_rho;
  in.n_queries = pl->ul.q_total;
  in.library_entries = pl->ul.lib_dbg_total;
  in.neighbour_entries = pl->ul.nbr_total;
  in.n_work_items = (int64_t)pl->ul.items.size();
  in.device_bytes = pl->ar.total;
  in.pair_count = pl->ul.pairs;
  in.flop_count = pl->ul.flops;
  in.brute_flop_count = pl->ul.brute_flops;
  in.brute_pair_count = pl->ul.brute_pairs;
  in.search_query_count = pl->ul.search_queries;
  in.table_query_count = pl->ul.table_queries;
  in.table_bytes = (pl->ul.table_elem() + sizeof(float) * (pl->ul.table_tv ? 2 : 1)) *
                   (size_t)pl->ul.table_total;
  // launches of one ccm_run: order, tables, sampler, one brute-force and one
  // table-scan kernel per E present, rho
  in.launches_per_run = 4 + pl->ul.table_groups();  // order, observed values, sampler, rho, tables
  in.launches_per_run += pl->ul.member_groups.empty() ? 0 : 1;  // membership words
  in.launches_per_run += pl->ul.tables.empty() ? 0 : 1;         // the tables' points
  in.launches_per_run += (int64_t)(pl->ul.groups.size() + pl->ul.groups_table.size());
  *out = pl.release();
  return CCM_OK;
}

ccm_status ccm_plan_get_info(const ccm_plan_t* plan, ccm_plan_info* info) {
  if (!plan || !info) return fail(CCM_EINVAL, "NULL argument");
  *info = plan->info;
  return CCM_OK;
}

ccm_status ccm_plan_destroy(ccm_plan_t* plan) {
  if (!plan) return fail(CCM_EINVAL, "plan is NULL");
  cudaSetDevice(plan->ctx->device);
  if (plan->stream) cudaStreamSynchronize(plan->stream);
  if (plan->graph) cudaGraphExecDestroy(plan->graph);
  if (plan->stream) cudaStreamDestroy(plan->stream);
  for (cudaEvent_t ev : plan->ev)
    if (ev) cudaEventDestroy(ev);
  cudaFree(plan->d_arena);
  release(plan->ctx, plan->ar.total);
  delete plan;
  return CCM_OK;
}

ccm_status ccm_run_ex(ccm_plan_t* plan, const float* series, double* rho, const ccm_debug_out* dbg,
                      void* cuda_stream) {
  if (!plan || !series || !rho) return fail(CCM_EINVAL, "NULL argument");
  std::lock_guard<std::mutex> g(plan->run_mu);
  CCM_CUDA(cudaSetDevice(plan->ctx->device));
  const ProblemCopy& pc = plan->pc;
  const bool in_dev = (pc.flags & CCM_INPUT_ON_DEVICE) != 0;
  const bool out_dev = (pc.flags & CCM_OUTPUT_ON_DEVICE) != 0;
  const size_t series_bytes = sizeof(float) * (size_t)pc.V * (size_t)pc.n;
  if (!in_dev && !all_finite(series, (size_t)pc.V * (size_t)pc.n))
    return fail(CCM_EINVAL, "series holds a non-finite value");
  cudaStream_t s = cuda_stream ? (cudaStream_t)cuda_stream : plan->stream;
  char* base = plan->d_arena;
  CCM_CUDA(cudaMemcpyAsync(base + plan->ar.series, series, series_bytes,
                           in_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
  const bool want_dbg = dbg && (dbg->libraries || dbg->neighbours || dbg->predictions);
  if (want_dbg) {
    // Checking path: direct launches with the per-unit outputs (no graph).
    const UnitList& ul = plan->ul;
    const size_t lb = sizeof(int32_t) * (size_t)ul.lib_dbg_total;
    const size_t nb = sizeof(int32_t) * (size_t)ul.nbr_total;
    const size_t xb = sizeof(float) * (size_t)ul.q_total;
    char* tmp = nullptr;
    if (!out_dev) {
      CCM_CUDA(cudaMallocAsync(&tmp, align_up(lb, 256) + align_up(nb, 256) + align_up(xb, 256), s));
    }
    int32_t* d_lib = dbg->libraries ? (out_dev ? dbg->libraries : reinterpret_cast<int32_t*>(tmp))
                                    : nullptr;
    int32_t* d_nbr = dbg->neighbours ? (out_dev ? dbg->neighbours
                                                : reinterpret_cast<int32_t*>(tmp + align_up(lb, 256)))
                                     : nullptr;
    float* d_xh = dbg->predictions
                      ? (out_dev ? dbg->predictions
                                 : reinterpret_cast<float*>(tmp + align_up(lb, 256) + align_up(nb, 256)))
                      : nullptr;
    ccm_status st =
        enqueue_sweep(base, plan->ar, ul, plan->tuning, plan->grid, plan->grid_table, plan->grid_scan, 1, d_lib,
                      d_nbr, d_xh, s, plan->ev, false, (pc.flags & CCM_SEARCH_STATS) != 0);
    if (st != CCM_OK) return st;
    if (!out_dev) {
      if (dbg->libraries) CCM_CUDA(cudaMemcpyAsync(dbg->libraries, d_lib, lb, cudaMemcpyDeviceToHost, s));
      if (dbg->neighbours) CCM_CUDA(cudaMemcpyAsync(dbg->neighbours, d_nbr, nb, cudaMemcpyDeviceToHost, s));
      if (dbg->predictions) CCM_CUDA(cudaMemcpyAsync(dbg->predictions, d_xh, xb, cudaMemcpyDeviceToHost, s));
      CCM_CUDA(cudaFreeAsync(tmp, s));
    }
  } else {
    if (!plan->tuned) {
      bool missing = false;
      for (int e = plan->ul.emin; e <= plan->ul.emax; ++e)
        for (const int32_t E : pc.E) missing |= (E == e && !plan->tuning.known[e]);
      if (missing && !(pc.flags & CCM_NO_AUTOTUNE) && plan->ul.pairs >= kTunePairs) {
        ccm_status st = autotune(plan, s);
        if (st != CCM_OK) return st;
      }
      plan->tuned = true;
    }
    if (!plan->graph) {
      cudaGraph_t graph = nullptr;
      TableBranch branch;  // (destroyed after the capture: the graph keeps the dependencies)
      const bool fork = !plan->ul.tables.empty() && plan->ul.max_nm <= kBranchMaxNm;
      if (fork) CCM_CUDA(branch.create());
      CCM_CUDA(cudaStreamBeginCapture(plan->stream, cudaStreamCaptureModeThreadLocal));
      ccm_status st = enqueue_sweep(base, plan->ar, plan->ul, plan->tuning, plan->grid,
                                    plan->grid_table, plan->grid_scan, 1, nullptr, nullptr, nullptr, plan->stream,
                                    plan->ev, true, (pc.flags & CCM_SEARCH_STATS) != 0,
                                    fork ? &branch : nullptr);
      const cudaError_t ce = cudaStreamEndCapture(plan->stream, &graph);
      if (st != CCM_OK) {
        if (graph) cudaGraphDestroy(graph);
        return st;
      }
      CCM_CUDA(ce);
      const cudaError_t ie = cudaGraphInstantiate(&plan->graph, graph, 0);
      cudaGraphDestroy(graph);
      CCM_CUDA(ie);
    }
    CCM_CUDA(cudaGraphLaunch(plan->graph, s));
  }
  const size_t rho_bytes = sizeof(double) * (size_t)plan->ul.n_rho;
  CCM_CUDA(cudaMemcpyAsync(rho, base + plan->ar.rho, rho_bytes,
                           out_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
  if (!cuda_stream || !in_dev || !out_dev) return check_err_flag(base, plan->ar, s);
  return CCM_OK;
}

ccm_status ccm_plan_kernel_times(const ccm_plan_t* plan, double* sampler_ms, double* knn_ms) {
  double st[4];
  const ccm_status r = ccm_plan_stage_times(plan, st);
  if (r != CCM_OK) return r;
  if (sampler_ms) *sampler_ms = st[0] + st[1];
  if (knn_ms) *knn_ms = st[2] + st[3];
  return CCM_OK;
}

ccm_status ccm_plan_stage_times(const ccm_plan_t* plan, double* stage_ms) {
  if (!plan || !stage_ms) return fail(CCM_EINVAL, "NULL argument");
  CCM_CUDA(cudaSetDevice(plan->ctx->device));
  const int from[4] = {0, 1, 2, 3}, to[4] = {5, 2, 3, 4};
  float t = 0.f;
  for (int q = 0; q < 4; ++q) {
    CCM_CUDA(cudaEventElapsedTime(&t, plan->ev[from[q]], plan->ev[to[q]]));
    stage_ms[q] = t;
  }
  CCM_CUDA(cudaEventElapsedTime(&t, plan->ev[5], plan->ev[4]));  // it also waits for the tables
  stage_ms[3] = std::min(stage_ms[3], (double)t);
  return CCM_OK;
}

ccm_status ccm_plan_search_stats(const ccm_plan_t* plan, ccm_search_stats* out) {
  if (!plan || !out) return fail(CCM_EINVAL, "NULL argument");
  if (!(plan->pc.flags & CCM_SEARCH_STATS))
    return fail(CCM_EINVAL, "the plan was made without CCM_SEARCH_STATS");
  CCM_CUDA(cudaSetDevice(plan->ctx->device));
  unsigned long long c[kStatCount];
  CCM_CUDA(cudaMemcpy(c, plan->d_arena + plan->ar.stats, sizeof(c), cudaMemcpyDeviceToHost));
  out->brute_tiles = c[kStatBruteTiles];
  out->brute_queries = c[kStatBruteQueries];
  out->pairs_begun = c[kStatPairsBegun];
  out->pairs_full = c[kStatPairsFull];
  out->pairs_pruned = c[kStatPairsPruned];
  out->candidates = c[kStatCandidates];
  out->merge_slots = c[kStatMergeSlots];
  out->table_queries = c[kStatTableQueries];
  out->table_entries = c[kStatTableEntries];
  out->table_fallbacks = c[kStatTableFallbacks];
  return CCM_OK;
}

ccm_status ccm_run(ccm_plan_t* plan, const float* series, double* rho, void* cuda_stream) {
  return ccm_run_ex(plan, series, rho, nullptr, cuda_stream);
}

ccm_status ccm_run_plain(ccm_plan_t* plan, const float* series, double* rho, void* cuda_stream) {
  if (!plan || !series || !rho) return fail(CCM_EINVAL, "NULL argument");
  std::lock_guard<std::mutex> g(plan->run_mu);
  CCM_CUDA(cudaSetDevice(plan->ctx->device));
  const ProblemCopy& pc = plan->pc;
  const bool in_dev = (pc.flags & CCM_INPUT_ON_DEVICE) != 0;
  const bool out_dev = (pc.flags & CCM_OUTPUT_ON_DEVICE) != 0;
  if (!in_dev && !all_finite(series, (size_t)pc.V * (size_t)pc.n))
    return fail(CCM_EINVAL, "series holds a non-finite value");
  cudaStream_t s = cuda_stream ? (cudaStream_t)cuda_stream : plan->stream;
  char* base = plan->d_arena;
  const Arena& ar = plan->ar;
  CCM_CUDA(cudaMemcpyAsync(base + ar.series, series, sizeof(float) * (size_t)pc.V * (size_t)pc.n,
                           in_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, s));
  CCM_CUDA(cudaMemsetAsync(base + ar.err, 0, sizeof(int32_t), s));
  SamplerParams sp = sampler_params(base, ar, plan->ul);
  sp.list_all = 1;
  const UnitDesc* d_units = reinterpret_cast<const UnitDesc*>(base + ar.units);
  const TargetDesc* d_targets = reinterpret_cast<const TargetDesc*>(base + ar.targets);
  CCM_CUDA(enqueue_order(base, ar, plan->ul, s));
  for (size_t q = 0; q < plan->ul.units.size(); ++q) {
    const UnitDesc& u = plan->ul.units[q];
    CCM_CUDA(launch_sampler(sp, (int64_t)q, 1, u.n_m, s));
    for (int32_t t = 0; t < u.n_targets; ++t)
      CCM_CUDA(launch_plain_unit(reinterpret_cast<const float*>(base + ar.series), d_units + q, u,
                                 d_targets + u.tgt_off + t,
                                 reinterpret_cast<const int32_t*>(base + ar.lib),
                                 reinterpret_cast<float*>(base + ar.scratch),
                                 reinterpret_cast<double*>(base + ar.rho), s));
  }
  CCM_CUDA(cudaMemcpyAsync(rho, base + ar.rho, sizeof(double) * (size_t)plan->ul.n_rho,
                           out_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s));
  if (!cuda_stream || !in_dev || !out_dev) return check_err_flag(base, ar, s);
  return CCM_OK;
}

ccm_status ccm_convergence(ccm_context* ctx, const double* rho, int64_t n_rows, int32_t n_L,
                           const int64_t* L, int32_t r, double z_crit,
                           ccm_convergence_t* out, uint32_t flags, void* cuda_stream) {
  static_assert(sizeof(ConvergenceRow) == sizeof(ccm_convergence_t), "layout");
  if (!ctx || !rho || !L || !out) return fail(CCM_EINVAL, "NULL argument");
  if (n_rows < 0 || n_rows > 0x7fffffff) return fail(CCM_EINVAL, "n_rows out of range");
  if (n_L < 2 || n_L > kMaxConvGroups) return fail(CCM_EINVAL, "n_L must be in 2..64");
  if (r < 1 || (int64_t)n_L * r > kMaxConvValues)
    return fail(CCM_EINVAL, "need r >= 1 and n_L*r <= 24576");
  if (std::isnan(z_crit)) return fail(CCM_EINVAL, "z_crit is NaN");
  ConvOrder ord;
  std::memset(&ord, 0, sizeof(ord));
  for (int32_t g = 0; g < n_L; ++g) ord.group[g] = g;
  std::stable_sort(ord.group, ord.group + n_L, [&](int32_t a, int32_t b) { return L[a] < L[b]; });
  for (int32_t g = 1; g < n_L; ++g)
    if (L[ord.group[g]] == L[ord.group[g - 1]]) return fail(CCM_EINVAL, "L values must differ");
  if (n_rows == 0) return CCM_OK;
  CCM_CUDA(cudaSetDevice(ctx->device));
  const bool in_dev = (flags & CCM_INPUT_ON_DEVICE) != 0;
  const bool out_dev = (flags & CCM_OUTPUT_ON_DEVICE) != 0;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const size_t rho_bytes = sizeof(double) * (size_t)n_rows * (size_t)n_L * (size_t)r;
  const size_t out_bytes = sizeof(ccm_convergence_t) * (size_t)n_rows;
  double* d_rho = const_cast<double*>(rho);
  ConvergenceRow* d_out = reinterpret_cast<ConvergenceRow*>(out);
  void* tmp = nullptr;
  if (!in_dev || !out_dev) {
    CCM_CUDA(cudaMalloc(&tmp, (in_dev ? 0 : rho_bytes + 256) + (out_dev ? 0 : out_bytes)));
    char* t = static_cast<char*>(tmp);
    if (!in_dev) {
      d_rho = reinterpret_cast<double*>(t);
      t += (rho_bytes + 255) / 256 * 256;
    }
    if (!out_dev) d_out = reinterpret_cast<ConvergenceRow*>(t);
  }
  cudaError_t e = cudaSuccess;
  if (!in_dev) e = cudaMemcpyAsync(d_rho, rho, rho_bytes, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = launch_convergence(d_rho, n_rows, n_L, r, ord, z_crit, d_out, s);
  if (e == cudaSuccess && !out_dev)
    e = cudaMemcpyAsync(out, d_out, out_bytes, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess && (tmp || !cuda_stream)) e = cudaStreamSynchronize(s);
  if (tmp) {
    const cudaError_t e2 = cudaFree(tmp);
    if (e == cudaSuccess) e = e2;
  }
  if (e != cudaSuccess) return fail(CCM_ECUDA, std::string("ccm_convergence: ") + cudaGetErrorString(e));
  return CCM_OK;
}

}  // extern "C"

// ================================================================ serving ===
struct Job {
  uint64_t ticket = 0;
  ProblemCopy pc;
  float* h_series = nullptr;  // pinned copy (from the context's pool)
  double* h_rho = nullptr;    // pinned result (from the context's pool)
  size_t series_bytes = 0, rho_bytes = 0;
  int64_t n_units = 0;
  size_t footprint = 0;
  double pairs = 0.0;  // query-library pairs: the job's cost
  int room = 0;        // room_of its layout
  enum State { kQueued, kRunning, kDone, kFailed, kCancelled } state = kQueued;
  ccm_status status = CCM_PENDING;
  std::string err;
  double t_submit = 0, t_start = 0, t_finish = 0;
};

struct Batch {
  ccm_context* ctx = nullptr;
  std::vector<std::shared_ptr<Job>> jobs;
  UnitList ul;
  Arena ar;
  char* d_arena = nullptr;
  int32_t* h_err = nullptr;
  void* h_meta = nullptr;  // pinned copy of units, items and order jobs for the async upload
  size_t meta_bytes = 0;
  cudaStream_t stream = nullptr;
  std::atomic<bool> finished{false};
};

namespace {

// Device footprint of a job; where it exceeds the budget, with less room.
size_t job_footprint(const ccm_context* ctx, const ProblemCopy& pc, double* pairs, int* room) {
  size_t total = 0;
  for (int attempt = 0; attempt < kRooms; ++attempt) {
    UnitList ul;
    append_units(pc, 0, 0, &ul, room_of(ctx, attempt));
    *pairs = ul.pairs;
    *room = attempt;
    total = layout((int64_t)pc.V * pc.n, ul, ul.n_rho, 0).total;
    if (total <= ctx->budget || barest(ul)) break;
  }
  return total;
}

void CUDART_CB on_batch_done(void* arg) {
  Batch* b = static_cast<Batch*>(arg);
  ccm_context* ctx = b->ctx;
  {
    std::lock_guard<std::mutex> g(ctx->mu);
    b->finished.store(true);
  }
  ctx->cv.notify_all();
}

// Launch one batch (called by the serving thread without ctx->mu held).
// `inject`: the fault-injection hook chose this batch; it fails after its
// arena and series uploads have been enqueued, like a failing CUDA call there.
ccm_status launch_batch(ccm_context* ctx, Batch* b, bool inject) {
  int64_t series_elems = 0, out = 0;
  for (auto& j : b->jobs) {
    append_units(j->pc, series_elems, out, &b->ul, room_of(ctx, j->room));
    series_elems += (int64_t)j->pc.V * j->pc.n;
    out += j->n_units;
  }
  sort_items(&b->ul);
  b->ar = layout(series_elems, b->ul, out, 0);
  CCM_CUDA(cudaMallocAsync(&b->d_arena, b->ar.total, b->stream));
  char* base = b->d_arena;
  int64_t so = 0;
  for (auto& j : b->jobs) {
    const size_t bytes = sizeof(float) * (size_t)j->pc.V * (size_t)j->pc.n;
    CCM_CUDA(cudaMemcpyAsync(base + b->ar.series + sizeof(float) * so, j->h_series, bytes,
                             cudaMemcpyHostToDevice, b->stream));
    so += (int64_t)j->pc.V * j->pc.n;
  }
  if (inject) return fail(CCM_ECUDA, "injected fault (CCM_FAULT_INJECT_BATCH): batch launch failed");
  // Descriptors go through pinned staging: a copy from pageable memory would
  // wait for earlier work on this (reused) stream.
  // (units, work items, order jobs, targets, table jobs, table work items,
  // observed-value jobs, series jobs, scan groups)
  constexpr int kMeta = 9;
  const void* src[kMeta] = {b->ul.units.data(),   b->ul.items.data(),  b->ul.orders.data(),
                            b->ul.targets.data(), b->ul.tables.data(), b->ul.items_table.data(),
                            b->ul.obs_jobs.data(),  b->ul.series_jobs.data(),
                            b->ul.member_groups.data()};
  const size_t len[kMeta] = {sizeof(UnitDesc) * b->ul.units.size(),
                             sizeof(WorkItem) * b->ul.items.size(),
                             sizeof(OrderJob) * b->ul.orders.size(),
                             sizeof(TargetDesc) * b->ul.targets.size(),
                             sizeof(TableJob) * b->ul.tables.size(),
                             sizeof(WorkItem) * b->ul.items_table.size(),
                             sizeof(ObsJob) * b->ul.obs_jobs.size(),
                             sizeof(SeriesJob) * b->ul.series_jobs.size(),
                             sizeof(MemberGroup) * b->ul.member_groups.size()};
  const size_t dst[kMeta] = {b->ar.units,  b->ar.items,       b->ar.orders,  b->ar.targets,
                             b->ar.tables, b->ar.items_table, b->ar.obs_jobs, b->ar.series_jobs,
                             b->ar.member_groups};
  b->meta_bytes = 0;
  for (int q = 0; q < kMeta; ++q) b->meta_bytes += len[q];
  b->h_meta = pinned_get(ctx, b->meta_bytes);
  if (!b->h_meta) return fail(CCM_ENOMEM, "pinned allocation failed");
  char* hm = static_cast<char*>(b->h_meta);
  for (int q = 0; q < kMeta; ++q) {
    if (len[q] == 0) continue;
    std::memcpy(hm, src[q], len[q]);
    CCM_CUDA(cudaMemcpyAsync(base + dst[q], hm, len[q], cudaMemcpyHostToDevice, b->stream));
    hm += len[q];
  }
  Tuning tn;
  {
    std::lock_guard<std::mutex> g(ctx->mu);
    tn = ctx->tuning;
  }
  ccm_status st =
      enqueue_sweep(base, b->ar, b->ul, tn, 0, 0, 0, 0, nullptr, nullptr, nullptr, b->stream);
  if (st != CCM_OK) return st;
  int64_t ro = 0;
  for (auto& j : b->jobs) {
    CCM_CUDA(cudaMemcpyAsync(j->h_rho, base + b->ar.rho + sizeof(double) * ro,
                             sizeof(double) * (size_t)j->n_units, cudaMemcpyDeviceToHost, b->stream));
    ro += j->n_units;
  }
  CCM_CUDA(cudaMemcpyAsync(b->h_err, base + b->ar.err, sizeof(int32_t), cudaMemcpyDeviceToHost,
                           b->stream));
  CCM_CUDA(cudaFreeAsync(b->d_arena, b->stream));
  b->d_arena = nullptr;  // freed in stream order: the error path must not free it again
  CCM_CUDA(cudaLaunchHostFunc(b->stream, on_batch_done, b));
  return CCM_OK;
}

// No CUDA call that may synchronise (cudaFreeHost, cudaMallocHost,
// cudaStreamSynchronize, ...) is made while ctx->mu is held: the host callback
// that marks a batch finished takes ctx->mu, and its stream cannot advance
// until it returns.
void serve(ccm_context* ctx) {
  cudaSetDevice(ctx->device);
  std::vector<int32_t*> to_free;
  std::unique_lock<std::mutex> lk(ctx->mu);
  for (;;) {
    // Retire finished batches.
    for (auto it = ctx->inflight.begin(); it != ctx->inflight.end();) {
      Batch* b = it->get();
      if (!b->finished.load()) {
        ++it;
        continue;
      }
      const double t = now_s();
      size_t bytes = 0;
      for (auto& j : b->jobs) {
        bytes += j->footprint;
        j->t_finish = t;
        if (*b->h_err != 0) {
          j->state = Job::kFailed;
          j->status = CCM_ECUDA;
          j->err = "kernel reported error flag " + std::to_string(*b->h_err);
        } else {
          j->state = Job::kDone;
          j->status = CCM_OK;
        }
      }
      ctx->used -= std::min(ctx->used, bytes);
      // cudaFreeHost may synchronise; a pending host callback of another batch
      // needs ctx->mu to finish, so free after releasing the lock.
      to_free.push_back(b->h_err);
      pinned_put(ctx, b->h_meta, b->meta_bytes);  // pool mutex only, no CUDA call
      it = ctx->inflight.erase(it);
      ctx->cv.notify_all();
    }
    if (!to_free.empty()) {
      lk.unlock();
      for (int32_t* ptr : to_free) pinned_put(ctx, ptr, sizeof(int32_t));
      to_free.clear();
      lk.lock();
      continue;  // state may have changed while unlocked
    }
    if (ctx->stop && ctx->inflight.empty()) break;
    // Admit queued jobs into a new batch while their footprints fit.
    if (!ctx->stop && !ctx->queue.empty() && (int)ctx->inflight.size() < ctx->max_inflight) {
      auto b = std::make_shared<Batch>();
      b->ctx = ctx;
      size_t bytes = 0;
      int64_t units = 0;
      double pairs = 0.0;
      // A batch takes queued jobs in order while they fit the free budget; a
      // large job runs alone, small ones are grouped up to batch_pairs.
      while (!ctx->queue.empty()) {
        auto& j = ctx->queue.front();
        if (j->state == Job::kCancelled) {
          ctx->queue.pop_front();
          continue;
        }
        if (ctx->used + bytes + j->footprint > ctx->budget) break;
        if (!b->jobs.empty() && (units + j->n_units > (int64_t)1 << 22 ||
                                 pairs + j->pairs > ctx->batch_pairs))
          break;
        bytes += j->footprint;
        units += j->n_units;
        pairs += j->pairs;
        b->jobs.push_back(j);
        ctx->queue.pop_front();
      }
      if (!b->jobs.empty()) {
        ctx->used += bytes;
        const double t = now_s();
        for (auto& j : b->jobs) {
          j->state = Job::kRunning;
          j->t_start = t;
        }
        b->stream = (pairs <= ctx->batch_pairs)
                        ? ctx->fast_streams[ctx->next_fast++ % ctx->fast_streams.size()]
                        : ctx->streams[ctx->next_stream++ % ctx->streams.size()];
        ctx->inflight.push_back(b);
        const bool inject = ctx->batches_launched++ == ctx->inject_batch;
        lk.unlock();
        b->h_err = static_cast<int32_t*>(pinned_get(ctx, sizeof(int32_t)));
        ccm_status st = b->h_err ? launch_batch(ctx, b.get(), inject)
                                 : fail(CCM_ENOMEM, "pinned allocation failed");
        lk.lock();
        if (st != CCM_OK) {
          // Nothing more will run for this batch once the stream drains.
          lk.unlock();
          cudaStreamSynchronize(b->stream);
          if (b->d_arena) cudaFree(b->d_arena);
          lk.lock();
          for (auto& j : b->jobs) {
            j->state = Job::kFailed;
            j->status = st;
            j->err = t_err;
            j->t_finish = now_s();
          }
          ctx->used -= std::min(ctx->used, bytes);
          if (b->h_err) to_free.push_back(b->h_err);
          pinned_put(ctx, b->h_meta, b->meta_bytes);
          ctx->inflight.remove(b);
          ctx->cv.notify_all();
        }
        continue;
      }
    }
    ctx->cv.wait_for(lk, std::chrono::milliseconds(50));
  }
}

ccm_status ensure_server(ccm_context* ctx) {
  std::lock_guard<std::mutex> g(ctx->mu);
  if (ctx->server_started) return CCM_OK;
  int least = 0, greatest = 0;
  CCM_CUDA(cudaDeviceGetStreamPriorityRange(&least, &greatest));
  for (int q = 0; q < ctx->max_inflight / 2; ++q) {
    cudaStream_t s;
    CCM_CUDA(cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, least));
    ctx->streams.push_back(s);
    CCM_CUDA(cudaStreamCreateWithPriority(&s, cudaStreamNonBlocking, greatest));
    ctx->fast_streams.push_back(s);
  }
  ctx->server = std::thread(serve, ctx);
  ctx->server_started = true;
  return CCM_OK;
}

void free_job(ccm_context* ctx, Job* j) {
  pinned_put(ctx, j->h_series, j->series_bytes);
  pinned_put(ctx, j->h_rho, j->rho_bytes);
  j->h_series = nullptr;
  j->h_rho = nullptr;
}

}  // namespace

extern "C" {

ccm_status ccm_submit(ccm_context* ctx, const ccm_problem* prob, const float* series,
                      uint64_t* ticket) {
  if (!ctx || !series || !ticket) return fail(CCM_EINVAL, "NULL argument");
  auto j = std::make_shared<Job>();
  ccm_status st = copy_problem(prob, &j->pc);
  if (st != CCM_OK) return st;
  if (j->pc.flags & (CCM_INPUT_ON_DEVICE | CCM_OUTPUT_ON_DEVICE))
    return fail(CCM_EINVAL, "ccm_submit takes host series and returns host rho");
  const size_t elems = (size_t)j->pc.V * (size_t)j->pc.n;
  if (!all_finite(series, elems)) return fail(CCM_EINVAL, "series holds a non-finite value");
  j->n_units = j->pc.n_units();
  j->footprint = job_footprint(ctx, j->pc, &j->pairs, &j->room);
  if (j->footprint > ctx->budget)
    return fail(CCM_ETOOLARGE, "job footprint " + std::to_string(j->footprint) +
                                   " B exceeds the context budget");
  CCM_CUDA(cudaSetDevice(ctx->device));
  st = ensure_server(ctx);
  if (st != CCM_OK) return st;
  j->series_bytes = sizeof(float) * elems;
  j->rho_bytes = sizeof(double) * (size_t)j->n_units;
  j->h_series = static_cast<float*>(pinned_get(ctx, j->series_bytes));
  j->h_rho = static_cast<double*>(pinned_get(ctx, j->rho_bytes));
  if (!j->h_series || !j->h_rho) {
    free_job(ctx, j.get());
    return fail(CCM_ENOMEM, "pinned allocation failed");
  }
  std::memcpy(j->h_series, series, sizeof(float) * elems);
  j->t_submit = now_s();
  {
    std::lock_guard<std::mutex> g(ctx->mu);
    j->ticket = ctx->next_ticket++;
    ctx->jobs[j->ticket] = j;
    ctx->queue.push_back(j);
  }
  ctx->cv.notify_all();
  *ticket = j->ticket;
  return CCM_OK;
}

ccm_status ccm_poll(ccm_context* ctx, uint64_t ticket, double* rho, int32_t timeout_ms) {
  if (!ctx) return fail(CCM_EINVAL, "context is NULL");
  std::unique_lock<std::mutex> lk(ctx->mu);
  auto it = ctx->jobs.find(ticket);
  if (it == ctx->jobs.end()) return fail(CCM_ENOTFOUND, "unknown ticket");
  std::shared_ptr<Job> j = it->second;
  auto finished = [&] {
    return j->state == Job::kDone || j->state == Job::kFailed || j->state == Job::kCancelled;
  };
  if (!finished() && timeout_ms > 0)
    ctx->cv.wait_for(lk, std::chrono::milliseconds(timeout_ms), finished);
  if (!finished()) return CCM_PENDING;
  ccm_status st = j->status;
  if (j->state == Job::kDone) {
    if (!rho) return fail(CCM_EINVAL, "rho is NULL");
    std::memcpy(rho, j->h_rho, sizeof(double) * (size_t)j->n_units);
  } else {
    t_err = j->err;
  }
  ctx->jobs.erase(it);
  lk.unlock();
  free_job(ctx, j.get());
  return st;
}

ccm_status ccm_cancel(ccm_context* ctx, uint64_t ticket) {
  if (!ctx) return fail(CCM_EINVAL, "context is NULL");
  std::lock_guard<std::mutex> g(ctx->mu);
  auto it = ctx->jobs.find(ticket);
  if (it == ctx->jobs.end()) return fail(CCM_ENOTFOUND, "unknown ticket");
  Job* j = it->second.get();
  if (j->state != Job::kQueued) return CCM_PENDING;
  j->state = Job::kCancelled;
  j->status = CCM_ECANCELLED;
  j->err = "cancelled";
  j->t_finish = now_s();
  ctx->cv.notify_all();
  return CCM_OK;
}

ccm_status ccm_job_times(ccm_context* ctx, uint64_t ticket, double* submit_s, double* start_s,
                         double* finish_s) {
  if (!ctx) return fail(CCM_EINVAL, "context is NULL");
  std::lock_guard<std::mutex> g(ctx->mu);
  auto it = ctx->jobs.find(ticket);
  if (it == ctx->jobs.end()) return fail(CCM_ENOTFOUND, "unknown ticket");
  Job* j = it->second.get();
  if (submit_s) *submit_s = j->t_submit;
  if (start_s) *start_s = j->t_start;
  if (finish_s) *finish_s = j->t_finish;
  return (j->state == Job::kDone || j->state == Job::kFailed || j->state == Job::kCancelled)
             ? CCM_OK
             : CCM_PENDING;
}

ccm_status ccm_context_destroy(ccm_context* ctx) {
  if (!ctx) return fail(CCM_EINVAL, "context is NULL");
  {
    std::lock_guard<std::mutex> g(ctx->mu);
    ctx->stop = true;
    for (auto& j : ctx->queue) {
      if (j->state == Job::kQueued) {
        j->state = Job::kCancelled;
        j->status = CCM_ECANCELLED;
      }
    }
    ctx->queue.clear();
  }
  ctx->cv.notify_all();
  if (ctx->server_started) ctx->server.join();
  cudaSetDevice(ctx->device);
  for (cudaStream_t s : ctx->streams) cudaStreamDestroy(s);
  for (cudaStream_t s : ctx->fast_streams) cudaStreamDestroy(s);
  for (auto& kv : ctx->jobs) free_job(ctx, kv.second.get());
  ctx->jobs.clear();
  for (void* ptr : ctx->pool_all) cudaFreeHost(ptr);
  delete ctx;
  return CCM_OK;
}

}  // extern "C"
