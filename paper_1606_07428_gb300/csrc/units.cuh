// Work units that warps take in order from a device counter.  Plain C++ but for take_unit, so that the arithmetic
// can be tested without a GPU.
#pragma once

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

#ifdef __CUDACC__
__device__ __forceinline__ unit_t take_unit(unit_t* counter) {
  unit_t u = 0;
  if ((threadIdx.x & 31) == 0) u = atomicAdd(counter, 1u);
  return __shfl_sync(0xffffffffu, u, 0);
}
#endif

}  // namespace rbs
