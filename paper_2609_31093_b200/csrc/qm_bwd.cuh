// Dense masked backward of the block-sparse attention, for sequences of which a row selects a fair share (App. B; the
// list-driven kernel in bsa_bwd_kernel.cuh serves the others).  Tiles of 128 consecutive rows (128 / G tokens x G heads of
// one KV head) against 64- or 128-key steps, only those some row of the tile selected; everything by contiguous TMA tile
// loads, no inverted lists, no fp32 accumulators in memory (but for split key blocks):
//
//   qm_bwd_prep_kernel  per row: -lse2 and -delta = -dO . O; selection bits per token and their union per 128-row tile
//   qm_bwd_kv_kernel    one item per 128 keys: S^T = K Q^T, dP^T = V dO^T -> P^T, dS^T over them in TMEM ->
//                       dV += P^T dO, dK += dS^T Q in TMEM over the tiles that selected any of the keys
//   qm_bwd_q_kernel     one item per one or two tiles: S = Q K^T, dP = dO V^T -> dS over S in TMEM -> dQ += dS K in TMEM
//
// Seven products instead of the list kernel's five, but no gathers and no reductions into memory.
//
// A product over a tile multiplies every row with every key, zero weights included, so what is not finite has to be kept from
// what did not select it.  Rows (their denominator or delta shows it): their queries and gradients count as zero in a step, and
// the keys they did select get NaN through the row's bias.  Keys: sums that are not finite become zero where no row selected
// the key, and rows of dQ that are not finite are computed again from their own leaves.
#pragma once

#include "pisa_common.cuh"
#include "query_major.cuh"

namespace pisa {
namespace qmb {

struct Args {
  const qm::Seq* seqs;       // null: uniform batch.  Seq: bits_off -> bits, up_off -> tbits, leaf_off -> stat, pyr_row = its number
  const qm::SeqOrder* order;
  int nseq;
  int lgC, lgG;
  int n_tiles, n_pairs, n_keys;   // work items of the three kernels
  int per;                   // tiles per item of the q kernel: 1 or 2
  // parts the rows of one key block are dealt out to (their sums meet in dk_acc / dv_acc): every row attends to the first
  // leaf, so the first block of a sequence has steps for all of its tiles and is divided further than the others
  int splits, splits0;
  uint32_t* bits;            // [Hkv][len][W] per sequence, W = ceil(M1 / 32)
  uint32_t* tbits;           // [Hkv][W][tiles] per sequence
  float2* stat;              // [Hkv][len][G] per sequence: (-lse * log2 e, -inf for a row without keys, NaN; -delta)
  int32_t* chain;            // [n_pairs] the q kernel's items, per CTA (each holds the one before it + 1)
  const __nv_bfloat16 *q, *k, *v;   // strides of the geometry, for rows that are computed again
  const int32_t* idx;
  const float* lse;
  const __nv_bfloat16* out;
  const __nv_bfloat16* dout;
  __nv_bfloat16* dq;         // element strides dq_s (b, n, h)
  long long dq_s[3];
  __nv_bfloat16* dk;         // dense [tokens][Hkv][d]
  __nv_bfloat16* dv;
  // fp32, zeroed; splits > 1: like dk, dv; else, with splits0 > 1, the first blocks only: [sequence][Hkv][128][d]
  float* dk_acc;
  float* dv_acc;
  int32_t* ctr;              // [2] next item of the kv and q kernels, zeroed by the preparation
  uint32_t* count;           // null or: (tile, 128-key block) steps, zero before the preparation
  Gate gate;
  int32_t* status;
};

__device__ __forceinline__ qm::Seq seq_of(const Geometry& geo, const Args& a, int b) {
  qm::Seq q;
  const long long W = (geo.M[1] + 31) >> 5;
  const int tpt = 128 >> a.lgG;
  q.cu = (long long)b * geo.N;
  q.leaf_off = q.cu * geo.Hkv * geo.G;
  q.up_off = (long long)b * geo.Hkv * ((geo.N + tpt - 1) / tpt) * W;
  q.bits_off = q.cu * geo.Hkv * W;
  q.tok = 0; q.batch = b; q.len = geo.N; q.pyr_row = b; q.row0 = 0; q.leaf0 = 0;
  return q;
}

struct Loc { qm::Seq q; int h, part, split; };   // part: tile, group of `per` tiles (last ones first) or 128-key block (first ones first)
enum { kTiles = 0, kPairs = 1, kKeys = 2 };
template <int WHICH>
__device__ __forceinline__ Loc locate(const Geometry& geo, const Args& a, int item) {
  Loc r;
  const int unit = (WHICH == kKeys) ? 128 : (WHICH == kPairs ? 128 * a.per : 128) >> a.lgG;    // tokens per part
  int local = item, units = geo.B * geo.Hkv, len = geo.N;
  if (a.seqs != nullptr) {
    auto first = [&](int i) { return WHICH == kTiles ? a.order[i].item0t : WHICH == kPairs ? a.order[i].item0 : a.order[i].item0k; };
    int lo = 0, hi = a.nseq;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (first(mid) <= item) lo = mid; else hi = mid;
    }
    r.q = a.seqs[a.order[lo].seq];
    local = item - first(lo);
    units = geo.Hkv;
    len = r.q.len;
  }
  int back, u;
  r.split = 0;
  if (WHICH == kKeys) {
    const int n0 = units * a.splits0, per = units * a.splits;
    const bool first = local < n0;
    back = first ? 0 : 1 + (local - n0) / per;
    u = first ? local : (local - n0) % per;
    const int sp = first ? a.splits0 : a.splits;
    r.split = u % sp;
    u /= sp;
  } else {
    back = local / units;
    u = local - back * units;
  }
  if (a.seqs == nullptr) r.q = seq_of(geo, a, u / geo.Hkv);
  r.h = u % geo.Hkv;
  r.part = (WHICH == kKeys) ? back : (len + unit - 1) / unit - 1 - back;
  return r;
}

}  // namespace qmb

int qm_bwd_splits(long long key_items);
int qm_bwd_splits0(long long tiles_of_longest, int splits);
int qm_bwd_tiles_per_item(long long tiles);
// the kernels, uniform or packed; tokens: extent of the token dimension of q, k, v, out, dout
int launch_qm_bwd(const Geometry& g, const qmb::Args& a, const void* q, const void* k, const void* v, long long tokens,
                  cudaStream_t s);

}  // namespace pisa
