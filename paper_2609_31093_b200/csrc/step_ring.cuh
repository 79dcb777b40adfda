// The ring through which a scheduler warp hands the steps of its work items to the other roles of a CTA.
#pragma once

#include "tc_utils.cuh"

namespace pisa {

// step flags: first / last step of an item; no more steps; an item without steps; << tile: the tile needs the step / it is
// the last step the tile needs
constexpr int kFirst = 1, kLast = 2, kEnd = 4, kEmpty = 8, kNeed0 = 16, kLast0 = 64;

constexpr int kStepRing = 8;
struct StepRing {
  uint64_t full[kStepRing], empty[kStepRing];
  int4 e[kStepRing];                                        // (item, unit, flags, -)
};
__device__ __forceinline__ void ring_init(StepRing& r, int readers) {
  for (int i = 0; i < kStepRing; ++i) { tc::mbar_init(&r.full[i], 1); tc::mbar_init(&r.empty[i], (uint32_t)readers); }
}
// scheduler: one more step (called by the whole warp)
__device__ __forceinline__ bool ring_push(StepRing& r, int& n, int4 e, volatile int* fail) {
  const int s = n % kStepRing, lane = threadIdx.x & 31;
  bool ok = n < kStepRing || tc::mbar_wait_bounded(&r.empty[s], (uint32_t)((n / kStepRing - 1) & 1));
  ok = __all_sync(0xffffffffu, ok && !*fail);
  if (!ok) { *fail = 1; return false; }
  if (lane == 0) { r.e[s] = e; tc::mbar_arrive(&r.full[s]); }
  __syncwarp();
  ++n;
  return true;
}
// the other roles: the next step, false at the end (called by the whole warp)
__device__ __forceinline__ bool ring_pop(StepRing& r, int& n, int4& e, volatile int* fail) {
  const int s = n % kStepRing, lane = threadIdx.x & 31;
  bool ok = tc::mbar_wait_bounded(&r.full[s], (uint32_t)((n / kStepRing) & 1));
  ok = __all_sync(0xffffffffu, ok);
  if (!ok) { *fail = 1; return false; }
  const int4 x = r.e[s];
  __syncwarp();
  if (lane == 0) tc::mbar_arrive(&r.empty[s]);
  // (the same in all lanes, and visibly so: loop bounds and descriptors depend on them)
  e.x = __shfl_sync(0xffffffffu, x.x, 0); e.y = __shfl_sync(0xffffffffu, x.y, 0); e.z = __shfl_sync(0xffffffffu, x.z, 0); e.w = 0;
  ++n;
  return (e.z & kEnd) == 0;
}

}  // namespace pisa
