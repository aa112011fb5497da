// Work units of the near corrections (mobility and magnetostatic operators).
#pragma once

#include <climits>

#include "common.cuh"

namespace rbs {

// Near correction.  For a near pair (target particle i, source particle j) the contribution of j's
// upsampled nodes is added and that of its base nodes (already in the smooth sum) removed.  Warps take the units
// of list_near_units from a counter.  A pair of 144-node particles is 688 sources against five units of
// targets, so one block per pair left most of the SMs idle on lists of a few hundred pairs and most of its threads idle
// where orders mix.
// base: with the base nodes; else the upsampled nodes alone (for sums that leave near sources out).
struct NearArgs {
  unit_t nunits;
  bool base;
  unit_t* counter;
  const NearUnitItem* units;
  const int2* near;
  const long long* offset;
  const int* nodes;
  const int* up_index;
  const long long* up_off;
};
struct NearUnit {
  int t0, t1;           // targets [t0, t1) of particle i that the unit holds, 32 at most
  long long ub, oj;     // first upsampled node and first base node of j
  int s0, s1, nup;      // sources [s0, s1): below nup upsampled nodes, then base nodes
};
__device__ __forceinline__ bool next_near_unit(const NearArgs& A, NearUnit& n) {
  const unit_t unit = take_unit(A.counter);
  if (unit >= A.nunits) return false;
  const NearUnitItem it = A.units[unit];
  const int2 pr = A.near[it.pair];
  const long long oi = A.offset[pr.x];
  n.t0 = (int)oi + it.t;
  n.t1 = min(n.t0 + 32, (int)oi + A.nodes[pr.x]);
  const int u = A.up_index[pr.y];
  n.ub = A.up_off[u];
  n.nup = (int)(A.up_off[u + 1] - n.ub);
  n.oj = A.offset[pr.y];
  const int total = n.nup + (A.base ? A.nodes[pr.y] : 0);
  const int step = ((total + it.parts - 1) / it.parts + 3) & ~3;
  n.s0 = min(total, it.part * step);
  n.s1 = min(total, n.s0 + step);
  return true;
}

// The units of the context's near list (its counter, d_unit[1], is zeroed by the caller or the weight kernels);
// blocks: as many 128-thread blocks as have a unit per warp.
inline Status near_args(Context& c, bool base, NearArgs& A, int& blocks) {
  A.base = base;
  const long long units = (long long)c.d_near_units.n;
  if (!units_fit(units)) return Status::Err(RBS_ENOMEM, "near correction: more than 2^32 work units");
  A.nunits = (unit_t)units;
  A.counter = c.d_unit.ptr + 1;
  A.units = c.d_near_units.ptr;
  A.near = c.d_near.ptr;
  A.offset = c.d_offset.ptr;
  A.nodes = c.d_nodes.ptr;
  A.up_index = c.d_up_index.ptr;
  A.up_off = c.d_up_off.ptr;
  blocks = (int)std::min<long long>((units + 3) / 4, INT_MAX);
  return Status::Ok();
}

}  // namespace rbs
