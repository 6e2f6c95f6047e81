// Walk of one query's row of a distance indexing table for up to 32
// realizations at once (not part of the public ABI).
//
// A warp owns the query and a lane a realization.  The row holds the query's
// nearest manifold points, nearest first, as positions of the query order.  In
// a step the lanes read 32 consecutive ranks (one coalesced access), look up
// the membership word of each (bit r: realization r's library holds the point)
// and transpose the 32 x 32 bits across the warp, so that every lane holds the
// members of its own realization among the 32 ranks.  A lane that still lacks
// neighbours records the step's mask (at most K records: each holds a member);
// the walk ends when every lane has K.
#pragma once

#include "bits.cuh"
#include "ccm_internal.h"

namespace ccm {

// row: the query's entries (`stride` of them, a multiple of 64); order, m, W
// (kGeneral): the query order, the query's manifold index and its exclusion
// window; mask, step: the lane's columns of K records, kStep apart.  `dense`:
// the first 32 ranks mostly suffice.  Returns the members met; `steps` the
// steps of 32 ranks taken.
template <int K, int kStep, typename Index, bool kGeneral>
__device__ __forceinline__ int group_walk(const Index* row, int stride, bool dense, bool mine,
                                          const uint32_t* words, const int32_t* order, int m, int W,
                                          const BitTranspose& tr, uint32_t* mask, uint16_t* step,
                                          int& steps) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  // lane l holds rank 31 - l of a step, so that the highest set bit of a
  // realization's mask is its nearest member
  const Index* ip = row + (31 - lane);
  const Index* const end = ip + stride;
  int got = 0, recs = 0, c = 0;
  auto lookup = [&](uint32_t x) {
    uint32_t word = words[x];
    if (kGeneral && W > 0 && word != 0u) {  // points inside the exclusion window
      const int l = order[x];
      if ((unsigned)l - (unsigned)m + (unsigned)W <= 2u * (unsigned)W) word = 0u;
    }
    return word;
  };
  auto record = [&](uint32_t members) {
    if (members != 0u && got < K) {
      mask[recs * kStep] = members;
      step[recs * kStep] = (uint16_t)c;
      ++recs;
      got += __popc(members);
    }
    ++c;
  };
  uint32_t xa = (uint32_t)__ldg(ip);
  if (dense) {  // 32 ranks a step
    for (;;) {
      const uint32_t wa = lookup(xa);
      ip += 32;
      const bool more = ip < end;
      if (more) xa = (uint32_t)__ldg(ip);
      record(tr(wa));
      if (!more || !__any_sync(kAll, mine && got < K)) break;
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
      if (!more || !__any_sync(kAll, mine && got < K)) break;
    }
  }
  steps = c;
  return got;
}

// The first K ranks of a lane whose walk met at least K members.
template <int K, int kStep>
__device__ __forceinline__ void first_ranks(const uint32_t* mask, const uint16_t* step,
                                            int (&rank)[K]) {
  uint32_t cur = mask[0];
  int base = step[0] * 32, rec = 0;
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (cur == 0u) {
      ++rec;
      cur = mask[rec * kStep];
      base = step[rec * kStep] * 32;
    }
    const int b = __clz(cur);
    cur ^= 0x80000000u >> b;
    rank[s] = base + b;
  }
}

}  // namespace ccm
