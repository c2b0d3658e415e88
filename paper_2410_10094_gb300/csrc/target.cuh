// Where a group's outputs go, resolved by a warp (shared by the accumulation kernels).
#pragma once

#include "launch.h"

namespace stc {

// resolve_target by the 32 lanes of one warp (every lane calls it): the output plan is copied a
// word per lane rather than word by word, and only when the group's problem differs from the
// previous group's (a single contraction copies it once), so a group's set-up costs at most one
// round of loads. t.prob must hold kNoProb before the warp's first call.
__device__ __forceinline__ void resolve_target_warp(const GroupArgs& a, u64 g, unsigned n, OutTarget& t) {
  const unsigned lane = lane_id();
  uint32_t p = 0;
  if (lane == 0 && a.gprob) p = a.gprob[g];
  p = __shfl_sync(0xffffffffu, p, 0);
  const bool fresh = t.prob != p;
  __syncwarp();  // every lane has read t.prob before lane 0 rewrites it
  if (!fresh && !a.gprob) {  // a single contraction's next group: only the row and the base differ
    if (lane == 0) {
      t.fx = g;
      t.zrow = g * t.FY;
      t.base = n ? atomicAdd(t.counter, (u64)n) : 0;
    }
    __syncwarp();
    return;
  }
  const BatchOut* bo = a.bout + p;
  if (fresh) {
    const u64* src = reinterpret_cast<const u64*>(&bo->op);
    u64* dst = reinterpret_cast<u64*>(&t.op);
    constexpr unsigned kWords = sizeof(OutPlan) / sizeof(u64);
    for (unsigned i = lane; i < kWords; i += 32) dst[i] = src[i];
  }
  if (lane == 0) {
    t.prob = p;
    const u64 FY = bo->FY;
    t.FY = FY;
    t.fx = a.gfk ? a.gfk[g] : g;
    t.zrow = t.fx * FY;
    t.counter = a.bnz + p;
    t.base = n ? atomicAdd(a.bnz + p, (u64)n) : 0;
    t.cap = bo->out_cap;
    t.coords = bo->coords;
    t.vals = bo->vals;
  }
  __syncwarp();
}

}  // namespace stc
