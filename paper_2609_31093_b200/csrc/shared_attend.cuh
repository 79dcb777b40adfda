// Attention over the leaves that many rows of a 128-row query tile selected (see shared_attend.cu): the query-major part of the
// list-driven attention.
#pragma once

#include "pisa_common.cuh"

namespace pisa {

// Per tile of 128 / G consecutive tokens of one (batch, KV head): its shared leaves and who selected them.
struct SharedPlan {
  int max_leaves;            // room per tile
  int words;                 // mask words per leaf: one bit per token of the tile
  int tiles;                 // tiles per sequence
  uint16_t* leaf;            // [BH][tiles][max_leaves] ascending
  uint32_t* mask;            // [BH][tiles][max_leaves][words]
  int32_t* count;            // [BH][tiles]
  uint32_t* taken;           // [BH][N] bit s: entry s of the token's idx row is served here (the lists leave it out)
  int32_t* chain;            // [BH * tiles] the attention kernel's items, per CTA (each holds the one before it + 1)
};

bool shared_attend_supported(const Geometry& g, int dtype);
// lays the plan out in `ws`; returns its bytes (ws may be null)
size_t shared_plan_layout(const Geometry& g, char* ws, SharedPlan* plan);
int launch_shared_plan(const Geometry& g, const int32_t* idx, const SharedPlan& plan, cudaStream_t s);
// stores every accumulator row (layouts of pv_ws_kernel); ctr: zero on entry
int launch_shared_attend(const Geometry& g, const void* q, const void* k, const void* v, const float* row_lse, float* o_acc,
                         const SharedPlan& plan, int32_t* ctr, int32_t* status, cudaStream_t s);

}  // namespace pisa
