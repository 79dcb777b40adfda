// Query-major kernels: dense scoring of nodes and leaves, one-thread-per-token selection, masked dense attention.
//
// The list-driven kernels (tensor_path.cu) pay per (token, block) pair: a gathered query row in, an fp32 row of
// reductions out.  Where a row's K blocks are a fair share of all blocks before it -- short sequences -- a dense tile
// of consecutive tokens is cheaper: contiguous TMA tile loads, no lists, no accumulator in memory.  A tile is 128 rows
// (128 / G tokens x G heads of one KV head); a step is 128 consecutive keys (or node summaries).
//
//   qm_score_kernel   S = Q K^T per step; per-head log-sum-exp of every leaf; group-summed scores of the nodes of the
//                     levels that can prune (their children are level rows of the pyramid, 128 per step)
//   qm_select_kernel  one THREAD per (KV head, token): walks the levels, Select_K by a sorting network in registers
//   qm_attend_kernel  S = Q K^T, P = exp(S - lse) where selected, O += P V over the steps some row of the tile selected
//
// The first two also serve long sequences (upper levels only), with the leaf level left to the list-driven scoring.
#pragma once

#include "pisa_common.cuh"

namespace pisa {
namespace qm {

// One sequence of a packed launch (sequence-major outputs); a uniform batch computes the same from its geometry.
struct Seq {
  long long cu;            // tokens of the sequences before it: its idx block starts at Hkv*K*cu, its lse block at Hq*cu
  long long leaf_off;      // its leaf table   [Hkv][len][M1 padded to 4][G] floats
  long long up_off;        // its node table   [Hkv][len][width of the pruning levels] floats
  long long bits_off;      // its selection bits [Hkv][len][ceil(M1/32)] words
  int tok, batch;          // TMA coordinates of its first token
  int len;
  int pyr_row;             // packed: row of the pyramid scratch its levels start at, level l = [Hkv][M_l] rows
  int row0, leaf0;         // packed: tokens / leaves of the launch's sequences before it
};
// work items of the packed launch: sequence, its first item (longest sequences first); the backward's: groups of tiles in
// item0, tiles in item0t, 128-key blocks in item0k
struct SeqOrder { int seq, item0, item0t, item0k; };

struct Args {
  const Seq* seqs;         // null: uniform batch
  const SeqOrder* order;
  int nseq;
  int n_items;             // (tiles, KV head) work items
  int tiles;               // tiles per work item: 1 or 2 (two share every load of keys and values)
  int lgC, lgg, lgG;
  int t0, t1;              // uniform: tokens [t0, t1) are scored and selected (tables hold those rows only)
  int want_leaf;           // score the leaves (whole sequences only)
  float* leaf;
  float* up;
  uint32_t* bits;
  int32_t* ctr;            // work-item counter of the attention kernel (zeroed by the selection)
  int32_t* status;
};

// nodes of level l >= 1 of a sequence of `len` tokens (ceil of ceil = ceil of the product: all powers of two)
__host__ __device__ __forceinline__ int level_nodes(int len, int lgC, int lgg, int l) {
  const int s = lgC + (l - 1) * lgg;
  return s >= 31 ? 1 : (int)(((long long)len + (1LL << s) - 1) >> s);
}
__host__ __device__ __forceinline__ int level_shift(int lgC, int lgg, int l) {
  const int s = lgC + (l - 1) * lgg;
  return s > 31 ? 31 : s;                                   // t < 2^31: a larger span just means ancestor 0
}
// highest level with more than K nodes (0: none; nothing can prune)
__host__ __device__ __forceinline__ int top_level(int len, int lgC, int lgg, int K) {
  int l = 0;
  while (level_nodes(len, lgC, lgg, l + 1) > K) ++l;
  return l;
}
// columns of one level in the node table: padded so that four nodes are one aligned vector
__host__ __device__ __forceinline__ int level_width(int nodes) { return (nodes + 3) & ~3; }
__host__ __device__ __forceinline__ int table_width(int len, int lgC, int lgg, int top) {
  int w = 0;
  for (int l = 2; l <= top; ++l) w += level_width(level_nodes(len, lgC, lgg, l));
  return w;
}

__device__ __forceinline__ Seq uniform_seq(const Geometry& geo, const Args& a, int b, int width) {
  Seq q;
  const long long rows = a.t1 - a.t0;
  q.cu = (long long)b * geo.N;
  q.leaf_off = (long long)b * geo.Hkv * geo.N * level_width(geo.M[1]) * geo.G;
  q.up_off = (long long)b * geo.Hkv * rows * width;
  q.bits_off = (long long)b * geo.Hkv * geo.N * ((geo.M[1] + 31) >> 5);
  q.tok = 0; q.batch = b; q.len = geo.N; q.pyr_row = 0; q.row0 = 0; q.leaf0 = 0;
  return q;
}

// work item -> (sequence, KV head, group of `tiles` tiles); the most expensive (last) ones come first
struct Tile { Seq q; int h, tile; };
__device__ __forceinline__ Tile locate(const Geometry& geo, const Args& a, int item, int tiles) {
  Tile r;
  const int tpt = (128 * tiles) >> a.lgG;
  if (a.seqs == nullptr) {
    const int units = geo.B * geo.Hkv;
    const int nt = (a.t1 - a.t0 + tpt - 1) / tpt, back = item / units, u = item - back * units;
    r.tile = a.t0 / tpt + nt - 1 - back;
    r.h = u % geo.Hkv;
    r.q = uniform_seq(geo, a, u / geo.Hkv, 0);
    return r;
  }
  int lo = 0, hi = a.nseq;                                  // last entry of `order` with item0 <= item
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (a.order[mid].item0 <= item) lo = mid; else hi = mid;
  }
  r.q = a.seqs[a.order[lo].seq];
  const int local = item - a.order[lo].item0;
  const int nt = (r.q.len + tpt - 1) / tpt, back = local / geo.Hkv;
  r.tile = nt - 1 - back;
  r.h = local - back * geo.Hkv;
  return r;
}

}  // namespace qm
}  // namespace pisa
