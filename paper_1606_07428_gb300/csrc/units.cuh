// Work units that warps take in order from a device counter.  Plain C++ but for take_unit, so that the arithmetic
// can be tested without a GPU.
#pragma once

#include <algorithm>
#include <vector>

#ifdef __CUDACC__
#define RBS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define RBS_HOST_DEVICE inline
#endif

namespace rbs {

// Every resident warp takes one more unit after the last, so a launch of nearly as many units as the counter holds
// would see it wrap and hand out the first ones again: kMaxUnits leaves 2^20, more than warps are ever resident.  32 bits
// because 64 cost the solves 1% (the divisions of unit_part); no list comes near: a work item holds up to 128 nodes.
using unit_t = unsigned;
constexpr long long kMaxUnits = 0xffffffffLL - (1 << 20);
inline bool units_fit(long long units) { return units <= kMaxUnits; }

struct UnitPart {
  unit_t item;  // work item
  int part;     // its run of targets
};
RBS_HOST_DEVICE UnitPart unit_part(unit_t unit, int per_item) {
  const unit_t item = unit / (unit_t)per_item;
  return {item, (int)(unit - item * (unit_t)per_item)};
}

// A unit of the near corrections: 32 targets (from node t of the target particle on) of a near pair against one of
// `parts` equal runs of its sources.
struct alignas(16) NearUnitItem {
  int pair, t, part, parts;
};
// The units of near pairs with the given numbers of target and source nodes, pair by pair.  Source runs: about 16 units
// per SM over the whole list, of at least 128 sources and at most about 512 (a unit of one p = 16 source particle, 2,656
// sources, would outlast a list of mixed orders); one run per target where `one_part` is set.  Every unit has targets and
// sources of its own: units cut by the largest particles of the context, empty for the others, cost a suspension with
// one p = 32 particle among 500 of p = 4 nine times its near corrections' time (2.39 and 0.27 ms a float32 apply).
inline std::vector<NearUnitItem> list_near_units(const std::vector<int>& targets, const std::vector<int>& sources,
                                                 int sm_count, bool one_part) {
  long long chunks = 0;
  for (int t : targets) chunks += (t + 31) / 32;
  chunks = std::max(1LL, chunks);
  const long long fill = (16LL * sm_count + chunks - 1) / chunks;
  std::vector<NearUnitItem> out;
  out.reserve((size_t)chunks);
  for (size_t k = 0; k < targets.size(); ++k) {
    const int parts =
        one_part ? 1 : (int)std::max((sources[k] + 511LL) / 512, std::min<long long>(fill, sources[k] / 128));
    for (int t = 0; t < targets[k]; t += 32)
      for (int p = 0; p < parts; ++p) out.push_back({(int)k, t, p, parts});
  }
  return out;
}

#ifdef __CUDACC__
__device__ __forceinline__ unit_t take_unit(unit_t* counter) {
  unit_t u = 0;
  if ((threadIdx.x & 31) == 0) u = atomicAdd(counter, 1u);
  return __shfl_sync(0xffffffffu, u, 0);
}
#endif

}  // namespace rbs
