// What the rows of a 128-row query tile share: the query-major part of the list-driven path (shared_plan.cu, shared_score.cu,
// shared_attend.cu).
//
// The list-driven kernels (tensor_path.cu) gather a query row, and the attention adds an fp32 row into memory, for every
// (token, block) pair.  Neighbouring tokens select much the same blocks -- the first, the previous and their own by rule
// (App. B), others because they are about the same thing -- and for those a dense product of the tile's 128 rows with the block
// is cheaper, whoever selected it.  A plan says which blocks enough of a tile's tokens selected, and who did; the inverted
// lists keep the rest.
#pragma once

#include "pisa_common.cuh"

namespace pisa {

constexpr int kSharedMax = 176;      // blocks of one tile's list, at most

// Per tile of 128 / G consecutive tokens of one (batch, KV head): its shared blocks and who selected them.
struct SharedPlan {
  int threshold;             // tokens of a tile that make a block shared
  int span;                  // tokens under a block
  int max_nodes;             // room per tile
  int words;                 // mask words per block: one bit per token of the tile
  int tiles;                 // tiles per sequence
  uint16_t* node;            // [BH][tiles][max_nodes] ascending
  uint32_t* mask;            // [BH][tiles][max_nodes][words] who selected it, or (one of the two is null)
  uint8_t* slot;             // [BH][tiles][max_nodes][128 / G] the block's place in the token's row, 255 = not selected
  int32_t* count;            // [BH][tiles]
  uint32_t* taken;           // [BH][N] bit s: entry s of the token's row is served here (the lists leave it out)
  int32_t* chain;            // [BH * tiles] the attention kernel's items, per CTA (each holds the one before it + 1)
};

bool shared_supported(const Geometry& g, int dtype, int blocks);
// rows: [BH, N, K] blocks of plan.span tokens, ascending, -1 padded.  always0: block 0 is shared whoever selected it.
int launch_shared_plan(const Geometry& g, const int32_t* rows, const SharedPlan& plan, bool always0, cudaStream_t s);

// leaves, masks: lays the attention's plan out in `ws`; returns its bytes (ws may be null)
size_t shared_attend_layout(const Geometry& g, char* ws, SharedPlan* plan);
// stores every accumulator row (layouts of pv_ws_kernel); ctr: zero on entry
int launch_shared_attend(const Geometry& g, const void* q, const void* k, const void* v, const float* row_lse, float* o_acc,
                         const SharedPlan& plan, int32_t* ctr, int32_t* status, cudaStream_t s);

// level-2 nodes, slots: the leaf scoring's plan
size_t shared_score_layout(const Geometry& g, char* ws, SharedPlan* plan);
// per-head LSE of every child leaf of the shared nodes into blk_lse [BH, N, K * g, G]; ctr: zero on entry
int launch_shared_score(const Geometry& g, const void* q, const void* k, float* blk_lse, const SharedPlan& plan, int32_t* ctr,
                        int32_t* status, cudaStream_t s);

}  // namespace pisa
