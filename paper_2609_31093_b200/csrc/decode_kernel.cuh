// Decoding step (Sec. 3.3 "Decoding", App. B "Decode cache"): one new token per sequence, one launch.
//
// A thread-block cluster of sixteen to two CTAs (by how many clusters the batch needs resident at once) serves one
// (batch, KV head):
//   1. levels L..2: all live nodes of the levels that can prune are scored up front, eight per warp and round spread over
//      the cluster (m16n8k16 fragments: the query heads are the 16 rows of A, the nodes' children the columns of B), their
//      scores stored into every CTA's shared memory; every CTA then walks the levels from there, all 256 threads ranking
//      the candidates (block_select).  Hierarchies with more live nodes than the table holds are scored level by level,
//      candidates only, by every CTA redundantly;
//   2. the leaf candidates (at most g*K blocks of C raw keys, the large read of the selection) are spread over the
//      cluster's warps, half a block each where there are warps enough, the next keys in flight while the current ones
//      are scored; scores or per-head partials go to every CTA's shared memory;
//   3. after a cluster barrier every CTA applies the same final selection;
//   4. attention over the selected blocks in pieces of 16 or 32 keys spread over the cluster's warps: logits on the same
//      fragments, softmax in the lanes that hold them, probabilities (fp32) through shared memory, P V on the FMA pipe
//      with the number of heads a template parameter;
//   5. partial (max, sum, output) are merged inside a CTA, then across the cluster through distributed shared memory, a
//      slice of the outputs per CTA.
// The cached pyramid is refreshed along the new tokens' paths by clusters of their own at the end of the grid, one warp per
// (batch, KV head): nothing in the same step reads those nodes (the path is forced, never scored).
// Cluster barriers are hardware barriers among co-scheduled CTAs: there is no software spin anywhere.
//
// What bounds it: latency (dependent loads per phase, two large reads).  In SM cycles at the headline shape, 128K context,
// batch 1: the walk took 24 K (6 K per level: a round trip for the candidates' children, one warp's sorting network), level
// by level with block_select 15 K; leaf scoring 10.5 K; attention 26 K in clusters of eight (sixteen predicated head
// iterations for G = 4, one lane per head in the softmax), 12 K with the heads a template parameter; and the refresh used
// to end 10 K after everything else.
#pragma once

#include <math_constants.h>

#include "launch.cuh"
#include "lse_chunk.cuh"
#include "mma_frag.cuh"
#include "pisa_common.cuh"

namespace pisa {

using namespace frag;

constexpr int kDecTabNodes = 4096;                  // scores the up-front scoring's table holds (16 KB)

struct DecArgs {
  int pos;                              // position of the new token
  int units;                            // (batch, KV head) pairs: clusters beyond them refresh the pyramid
  int l_top, n_init;                    // level of the first candidate list (the nodes 0 .. n_init - 1)
  int anc[kMaxLevels], prev[kMaxLevels];   // ancestors of the current / previous leaf, [1] = the leaves themselves
  int n_tiles;                          // rounds of eight nodes of the up-front scoring (0: level by level)
  int tile0[kMaxLevels];                // ... first round of level l; its nodes' scores start at 8 * tile0[l] of the table
  const __nv_bfloat16* q;               // [B, Hq, d]
  const __nv_bfloat16* k;               // caches [B, Ncap, Hkv, d] (strides from the geometry)
  const __nv_bfloat16* v;
  __nv_bfloat16* pyr;                   // cached pyramid, capacity layout
  int32_t* idx;                         // [B, Hkv, K]
  __nv_bfloat16* out;                   // [B, Hq, d]
  float* lse;                           // [B, Hq]
};

namespace {

constexpr int kDecWarps = 8;
constexpr int kDecThreads = kDecWarps * 32;

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// address of `p` (this CTA's shared memory) in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t remote_smem(const void* p, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ float ld_remote(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}

// One logit into a candidate's running score state (Sec. 4.3).  LSE score: (m, acc) = running max and sum of
// exponentials.  Moment scores: m = the shift, acc and sq = first and second moments about it.
__device__ __forceinline__ void score_add(int mode, float& m, float& acc, float& sq, float z) {
  if (mode == PISA_SCORE_LSE) lse_add(m, acc, z);
  else { const float dl = z - m; acc += dl; sq += dl * dl; }
}
__device__ __forceinline__ float score_finish(int mode, float m, float acc, float sq, int n) {
  if (mode == PISA_SCORE_LSE) return m + __logf(acc);
  const float mu = acc / (float)n;
  return m + mu + ((mode == PISA_SCORE_MEAN_VAR) ? 0.5f * fmaxf(sq / (float)n - mu * mu, 0.f) : 0.f);
}

// The group's query heads as A fragments: row = head (zero beyond G; rows 8..15 only when WIDE), contraction index
// permuted so that a lane's pieces of a B row are contiguous 16-byte chunks (see mma_frag.cuh)
template <int D, bool WIDE>
struct HeadFrag {
  uint4 lo[D / 32], hi[WIDE ? D / 32 : 1];
  __device__ __forceinline__ void load(const __nv_bfloat16* q, int G, int lane) {
    const int gid = lane >> 2, tig = lane & 3;
    const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
    for (int c4 = 0; c4 < D / 32; ++c4) {
      lo[c4] = (gid < G) ? ldg128(q + gid * D + (c4 * 4 + tig) * 8) : zero;
      if constexpr (WIDE) hi[c4] = (gid + 8 < G) ? ldg128(q + (gid + 8) * D + (c4 * 4 + tig) * 8) : zero;
    }
  }
};
// one row of B per lane group: row gid of eight rows
template <int D>
struct RowFrag {
  uint4 w[D / 32];
  __device__ __forceinline__ void load(const __nv_bfloat16* row, bool ok, int lane) {
    const int tig = lane & 3;
#pragma unroll
    for (int c4 = 0; c4 < D / 32; ++c4) w[c4] = ok ? ldg128(row + (c4 * 4 + tig) * 8) : make_uint4(0u, 0u, 0u, 0u);
  }
};
// z[0..1] = head gid . rows 2*tig, 2*tig + 1;  z[2..3] = head gid + 8 . same rows
template <int D, bool WIDE>
__device__ __forceinline__ void heads_dot(const HeadFrag<D, WIDE>& q, const RowFrag<D>& r, float (&z)[4]) {
  z[0] = z[1] = z[2] = z[3] = 0.f;
#pragma unroll
  for (int c4 = 0; c4 < D / 32; ++c4) {
    mma_bf16_16816(z, q.lo[c4].x, WIDE ? q.hi[WIDE ? c4 : 0].x : 0u, q.lo[c4].y, WIDE ? q.hi[WIDE ? c4 : 0].y : 0u, r.w[c4].x, r.w[c4].y);
    mma_bf16_16816(z, q.lo[c4].z, WIDE ? q.hi[WIDE ? c4 : 0].z : 0u, q.lo[c4].w, WIDE ? q.hi[WIDE ? c4 : 0].w : 0u, r.w[c4].z, r.w[c4].w);
  }
}

// Select_K among n <= 128 candidates by all 256 threads: every candidate's rank under (score descending, position
// ascending) is counted by four (n <= 64) or two threads, the kept ones (all of them when n <= K) are handed, in order, to
// emit(position, candidate).  u: scores (rankable), 16-byte aligned, -inf from n to the next multiple of 64 when n > K.
// Returns the number kept.  Starts and ends with a barrier.
template <typename Emit>
__device__ __forceinline__ int block_select(const float* u, int n, int K, int* s_cnt, Emit&& emit) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  __syncthreads();
  if (n <= K) {
    if (tid < n) emit(tid, tid);
    __syncthreads();
    return n;
  }
  const int lg = (n <= 64) ? 2 : 1, s = tid >> lg, part = tid & ((1 << lg) - 1);
  const int seg = (n <= 64) ? 4 : 16;                       // vectors of four scores per thread
  const float ui = u[s];
  const float4* u4 = reinterpret_cast<const float4*>(u) + part * seg;
  int rank = 0;
#pragma unroll 4
  for (int j = 0; j < seg; ++j) {
    const float4 x = u4[j];
    const int j0 = (part * seg + j) * 4;
    rank += (x.x > ui || (x.x == ui && j0 < s)) + (x.y > ui || (x.y == ui && j0 + 1 < s)) +
            (x.z > ui || (x.z == ui && j0 + 2 < s)) + (x.w > ui || (x.w == ui && j0 + 3 < s));
  }
  rank += __shfl_xor_sync(0xffffffffu, rank, 1);
  if (lg == 2) rank += __shfl_xor_sync(0xffffffffu, rank, 2);
  const bool keep = part == 0 && s < n && rank < K;
  const unsigned bal = __ballot_sync(0xffffffffu, keep);
  if (lane == 0) s_cnt[warp] = __popc(bal);
  __syncthreads();
  int base = 0;
#pragma unroll
  for (int w = 0; w < kDecWarps; ++w) base += (w < warp) ? s_cnt[w] : 0;
  if (keep) emit(base + __popc(bal & ((1u << lane) - 1u)), s);
  __syncthreads();
  return K;
}

// The new token's path in the cached pyramid, by one warp (lane = d / 32 columns): the current leaf's mean over the keys it
// holds so far, recomputed from the raw keys, then each ancestor's over its stored children.  The siblings on the path are
// read up front (kSibLevels levels of them), so that the dependent part is arithmetic.
template <int D>
__device__ void refresh_path(const Geometry& geo, const DecArgs& a, int b, int h, int lane) {
  constexpr int DV = D / 32, kSibLevels = 16;
  const int c = a.anc[1], t0 = c * geo.C, cnt = a.pos - t0 + 1;
  const long long bh = (long long)b * geo.Hkv + h;
  const __nv_bfloat16* kb = a.k + (long long)b * geo.ks[0] + (long long)h * geo.ks[2] + (long long)t0 * geo.ks[1] + lane * DV;
  auto load = [&](const __nv_bfloat16* p, float (&x)[DV]) {
    if constexpr (DV == 4) {
      const uint2 r = *reinterpret_cast<const uint2*>(p);
      x[0] = __uint_as_float(r.x << 16); x[1] = __uint_as_float(r.x & 0xFFFF0000u);
      x[2] = __uint_as_float(r.y << 16); x[3] = __uint_as_float(r.y & 0xFFFF0000u);
    } else {
      const uint32_t r = *reinterpret_cast<const uint32_t*>(p);
      x[0] = __uint_as_float(r << 16); x[1] = __uint_as_float(r & 0xFFFF0000u);
    }
  };
  auto siblings = [&](int l, float (&x)[DV]) {             // sum of the stored children of the path's level-l node before the path
#pragma unroll
    for (int j = 0; j < DV; ++j) x[j] = 0.f;
    const __nv_bfloat16* bl = a.pyr + geo.level_off[l - 1] + bh * geo.M[l - 1] * D + lane * DV;
    for (int r = a.anc[l] * geo.g; r < a.anc[l - 1]; ++r) {
      float y[DV];
      load(bl + (long long)r * D, y);
#pragma unroll
      for (int j = 0; j < DV; ++j) x[j] += y[j];
    }
  };
  float sib[kSibLevels][DV];
#pragma unroll
  for (int i = 0; i < kSibLevels; ++i)
    if (i + 2 <= geo.L) siblings(i + 2, sib[i]);
  float sum[DV];
#pragma unroll
  for (int j = 0; j < DV; ++j) sum[j] = 0.f;
  for (int r0 = 0; r0 < cnt; r0 += 16) {
    float x[16][DV];
#pragma unroll
    for (int u = 0; u < 16; ++u) {
#pragma unroll
      for (int j = 0; j < DV; ++j) x[u][j] = 0.f;
      if (r0 + u < cnt) load(kb + (long long)(r0 + u) * geo.ks[1], x[u]);
    }
#pragma unroll
    for (int u = 0; u < 16; ++u)
#pragma unroll
      for (int j = 0; j < DV; ++j) sum[j] += x[u][j];
  }
  float cur[DV];
  auto store = [&](int l, int node) {
    __nv_bfloat16* dst = a.pyr + geo.level_off[l] + (bh * geo.M[l] + node) * D + lane * DV;
#pragma unroll
    for (int j = 0; j < DV; j += 2) {
      const __nv_bfloat162 y = __floats2bfloat162_rn(sum[j], sum[j + 1]);
      *reinterpret_cast<__nv_bfloat162*>(dst + j) = y;
      cur[j] = __low2float(y); cur[j + 1] = __high2float(y);
    }
  };
#pragma unroll
  for (int j = 0; j < DV; ++j) sum[j] = sum[j] / (float)cnt;
  store(1, c);
  auto level = [&](int l, const float (&x)[DV]) {
    const float n = (float)(a.anc[l - 1] - a.anc[l] * geo.g + 1);            // valid children up to the path's
#pragma unroll
    for (int j = 0; j < DV; ++j) sum[j] = (x[j] + cur[j]) / n;
    store(l, a.anc[l]);
  };
#pragma unroll
  for (int i = 0; i < kSibLevels; ++i)
    if (i + 2 <= geo.L) level(i + 2, sib[i]);
  for (int l = kSibLevels + 2; l <= geo.L; ++l) {
    float x[DV];
    siblings(l, x);
    level(l, x);
  }
}

// the same as a launch of its own, for batches whose refreshing clusters do not fit into the step's grid (a third index
// there, read by every CTA, cost 0.4 us of the 34 of a step of 32 sequences)
template <int D>
__global__ void __launch_bounds__(kDecThreads) decode_refresh_kernel(const __grid_constant__ Geometry geo, const __grid_constant__ DecArgs a) {
  grid_dependency();
  const int u = blockIdx.x * kDecWarps + (threadIdx.x >> 5);
  if (u < a.units) refresh_path<D>(geo, a, u / geo.Hkv, u % geo.Hkv, threadIdx.x & 31);
}

// NG: query heads per KV head.  KT: keys per attention piece.  MINB = 1: all registers to one CTA per SM (lowest latency);
// MINB = 2: two CTAs per SM so that the latency-bound phases of different clusters overlap once the grid exceeds the SM
// count.  CLU: CTAs per cluster.  MOM: false = LSE score, true = the mean / mean + variance scores.
template <int D, int NG, int KT, int MINB, int CLU, bool MOM>
__global__ void __cluster_dims__(CLU, 1, 1) __launch_bounds__(kDecThreads, MINB)
decode_step_kernel(const __grid_constant__ Geometry geo, const __grid_constant__ DecArgs a) {
  constexpr bool WIDE = NG > 8;
  constexpr int DV = D / 32;                               // output columns per lane
  constexpr int W = NG * D + 2 * NG;                       // floats per partial: o[NG][D], m[NG], l[NG]
  constexpr int PARTS = (!MOM && CLU >= 8) ? 2 : 1;        // a leaf may be scored by two warps
  extern __shared__ __align__(16) float s_dyn[];           // [kDecWarps][W] warp partials, [W] the CTA's; before that, leaf partials
  __shared__ float s_tab[kDecTabNodes];
  __shared__ int s_cand[2][kMaxCand];
  __shared__ __align__(16) float s_u[kMaxCand], s_leaf[kMaxCand];
  __shared__ int s_sel[kMaxK], s_cnt[kDecWarps];
  __shared__ __align__(16) float s_p[kDecWarps][KT][NG];   // per warp: probabilities [key][head]
  __shared__ __align__(16) float s_alpha[kDecWarps][NG];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gid = lane >> 2, tig = lane & 3;
  const int rank = blockIdx.x;                            // cluster spans the x dimension
  const int bh = blockIdx.y;
  grid_dependency();
  if (bh >= a.units) {                                    // a refreshing cluster: none of its CTAs meets a cluster barrier
    const int u = ((bh - a.units) * CLU + rank) * kDecWarps + warp;
    if (u < a.units) refresh_path<D>(geo, a, u / geo.Hkv, u % geo.Hkv, lane);
    return;
  }
  const int b = bh / geo.Hkv, h = bh % geo.Hkv;
  const int K = geo.K, g = geo.g, C = geo.C;
  const int mode = MOM ? geo.score_mode : (int)PISA_SCORE_LSE;
  const int pos = a.pos, c = a.anc[1];

  cluster_arrive();                                       // (distributed shared memory needs every CTA to have started)
  HeadFrag<D, WIDE> qf;
  qf.load(a.q + ((long long)b * geo.Hq + (long long)h * NG) * D, NG, lane);

  // ---------------------------------------------------------------- 1. levels L..2
  // group-summed scores of eight nodes by this warp: lane group gid takes `node`'s children as columns; afterwards every
  // lane holds the scores of nodes 2 * tig and 2 * tig + 1 of the eight
  const int gw = rank * kDecWarps + warp;                  // warp of the cluster
  auto score_eight = [&](int l, int node, bool scored, float (&us)[2]) {
    const __nv_bfloat16* child = a.pyr + geo.level_off[l - 1] + (long long)bh * geo.M[l - 1] * D + (scored ? (long long)node * g * D : 0);
    float m[2][2], ssum[2][2], sq[2][2];                  // [head half][node 2*tig + x]
#pragma unroll
    for (int x = 0; x < 4; ++x) { m[x >> 1][x & 1] = -CUDART_INF_F; ssum[x >> 1][x & 1] = 0.f; sq[x >> 1][x & 1] = 0.f; }
    for (int r0 = 0; r0 < g; r0 += 2) {
      RowFrag<D> ra, rb;
      ra.load(child + (long long)r0 * D, scored, lane);
      rb.load(child + (long long)(r0 + 1) * D, scored && r0 + 1 < g, lane);
      float za[4], zb[4];
      heads_dot<D, WIDE>(qf, ra, za);
      heads_dot<D, WIDE>(qf, rb, zb);
#pragma unroll
      for (int x = 0; x < (WIDE ? 4 : 2); ++x) {
        float& mm = m[x >> 1][x & 1];
        if (mode != PISA_SCORE_LSE && r0 == 0) mm = za[x] * geo.scale;               // shift: the first child
        score_add(mode, mm, ssum[x >> 1][x & 1], sq[x >> 1][x & 1], za[x] * geo.scale);
        if (r0 + 1 < g) score_add(mode, mm, ssum[x >> 1][x & 1], sq[x >> 1][x & 1], zb[x] * geo.scale);
      }
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      us[x] = (gid < NG) ? score_finish(mode, m[0][x], ssum[0][x], sq[0][x], g) : 0.f;
      if (WIDE) us[x] += (gid + 8 < NG) ? score_finish(mode, m[1][x], ssum[1][x], sq[1][x], g) : 0.f;
      us[x] += __shfl_xor_sync(0xffffffffu, us[x], 4);
      us[x] += __shfl_xor_sync(0xffffffffu, us[x], 8);
      us[x] += __shfl_xor_sync(0xffffffffu, us[x], 16);
    }
  };
  const bool upfront = a.n_tiles > 0;
  if (upfront) {
    bool waited = false;
    for (int ti = gw; ti < a.n_tiles; ti += CLU * kDecWarps) {
      int l = 2;
      while (l < a.l_top && ti >= a.tile0[l + 1]) ++l;
      const int node = (ti - a.tile0[l]) * 8 + gid;
      float us[2];
      score_eight(l, node, node < a.anc[l], us);           // (nodes before the path's: all their children exist)
      if (!waited) { cluster_wait(); waited = true; }
      const int j = lane & 7;                              // this lane stores node j of the round into every fourth CTA
      const float v0 = __shfl_sync(0xffffffffu, us[0], j >> 1), v1 = __shfl_sync(0xffffffffu, us[1], j >> 1);
      for (int r = lane >> 3; r < CLU; r += 4) st_remote(remote_smem(&s_tab[ti * 8 + j], r), (j & 1) ? v1 : v0);
    }
    __syncwarp();
    if (!waited) cluster_wait();
    cluster_arrive();
  }
  // Levels whose live nodes (those that do not start after the query's leaf) number at most K keep everything, so the walk
  // starts at the highest level that has more, with every child of the live nodes of the level above as its candidates.
  int n = a.n_init, cur = 0;
  for (int s = tid; s < n; s += kDecThreads) s_cand[0][s] = s;
  if (upfront) cluster_wait();
  __syncthreads();
  for (int l = a.l_top; l >= 2; --l) {
    const int* cand = s_cand[cur];
    int* next = s_cand[cur ^ 1];
    const int anc = a.anc[l];
    const int nV = n - max(0, cand[n - 1] - anc);         // candidates are ascending; those past the path's node end the list
    const int nEnd = nV - 1 - (a.prev[l] != anc);         // scored: 1 .. nEnd - 1 (the others are forced); all their children exist
    if (nV > K) {
      if (upfront) {
        if (tid < kMaxCand)
          s_u[tid] = (tid >= nV) ? -CUDART_INF_F : (tid > 0 && tid < nEnd) ? rankable(s_tab[a.tile0[l] * 8 + cand[tid]]) : forced_score(tid);
      } else {
        for (int s = nV + tid; s < kMaxCand; s += kDecThreads) s_u[s] = -CUDART_INF_F;
        for (int k0 = warp * 8; k0 < nV; k0 += kDecThreads / 4) {
          const int kap = k0 + gid;
          const bool scored = kap > 0 && kap < nEnd;
          float us[2];
          score_eight(l, scored ? cand[kap] : 0, scored, us);
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const int s = k0 + 2 * tig + x;
            if (gid == 0 && s < nV) s_u[s] = (s > 0 && s < nEnd) ? rankable(us[x]) : forced_score(s);
          }
        }
      }
    }
    const int kept = block_select(s_u, nV, K, s_cnt, [&](int p, int s) {
      const int i = cand[s];
      for (int r = 0; r < g; ++r) next[p * g + r] = i * g + r;
    });
    n = kept * g;
    cur ^= 1;
  }

  // ---------------------------------------------------------------- 2. leaf candidates
  const int* cand = s_cand[cur];
  const int nV = n - max(0, cand[n - 1] - c);
  const int nEnd = nV - 1 - (a.prev[1] != c);
  const __nv_bfloat16* kbh = a.k + (long long)b * geo.ks[0] + (long long)h * geo.ks[2];
  const __nv_bfloat16* vbh = a.v + (long long)b * geo.vs[0] + (long long)h * geo.vs[2];
  if (!upfront) cluster_wait();
  const int n_sc = nV > K ? nEnd - 1 : 0;                   // leaves to score: candidates 1 .. nEnd - 1
  // two warps per leaf where the cluster has enough of them
  const int parts = (PARTS == 2 && 2 * n_sc <= CLU * kDecWarps && C >= 64) ? 2 : 1;
  if (n_sc > 0) {
    for (int s = tid; s < kMaxCand; s += kDecThreads)      // forced ones and the padding; the cluster's warps write the scores
      if (s < 1 || s >= nEnd) s_leaf[s] = (s < nV) ? forced_score(s) : -CUDART_INF_F;
    const int nk = C / parts;                              // keys per warp
    for (int w = gw; w < n_sc * parts; w += CLU * kDecWarps) {
      const int ci = 1 + (parts == 2 ? w >> 1 : w), pt = (parts == 2) ? w & 1 : 0;
      // a scored leaf lies strictly before the current one: all C keys exist and are visible
      const __nv_bfloat16* kl = kbh + ((long long)cand[ci] * C + pt * nk + gid) * geo.ks[1];
      const long long s8 = 8 * geo.ks[1];
      float m[2], ssum[2], sq[2];
      m[0] = m[1] = -CUDART_INF_F; ssum[0] = ssum[1] = 0.f; sq[0] = sq[1] = 0.f;
      constexpr int AHEAD = (MINB == 1 && !WIDE) ? 3 : 2;  // sixteen-key tiles in registers: this one and the next ones in flight
      RowFrag<D> r[AHEAD][2];
#pragma unroll
      for (int x = 0; x < AHEAD - 1; ++x) {
        r[x][0].load(kl + 2 * x * s8, 16 * x < nk, lane);
        r[x][1].load(kl + (2 * x + 1) * s8, 16 * x < nk, lane);
      }
      for (int kt = 0; kt < nk; kt += 16) {
        const __nv_bfloat16* kn = kl + (long long)(kt / 8 + 2 * (AHEAD - 1)) * s8;
        const bool more = kt + 16 * (AHEAD - 1) < nk;
        r[AHEAD - 1][0].load(kn, more, lane);
        r[AHEAD - 1][1].load(kn + s8, more, lane);
        float za[4], zb[4];
        heads_dot<D, WIDE>(qf, r[0][0], za);
        heads_dot<D, WIDE>(qf, r[0][1], zb);
#pragma unroll
        for (int x = 0; x < (WIDE ? 2 : 1); ++x) {
          const float y0 = za[2 * x] * geo.scale, y1 = za[2 * x + 1] * geo.scale, y2 = zb[2 * x] * geo.scale, y3 = zb[2 * x + 1] * geo.scale;
          if (mode == PISA_SCORE_LSE) {
            const float mn = fmaxf(m[x], fmaxf(fmaxf(y0, y1), fmaxf(y2, y3)));
            ssum[x] = ssum[x] * __expf(m[x] - mn) + ((__expf(y0 - mn) + __expf(y1 - mn)) + (__expf(y2 - mn) + __expf(y3 - mn)));
            m[x] = mn;
          } else {
            // moment scores: every lane of a head shifts by the logit of the block's first key
            if (kt == 0) m[x] = __shfl_sync(0xffffffffu, y0, lane & ~3);
            score_add(mode, m[x], ssum[x], sq[x], y0);
            score_add(mode, m[x], ssum[x], sq[x], y1);
            score_add(mode, m[x], ssum[x], sq[x], y2);
            score_add(mode, m[x], ssum[x], sq[x], y3);
          }
        }
#pragma unroll
        for (int x = 0; x < AHEAD - 1; ++x) { r[x][0] = r[x + 1][0]; r[x][1] = r[x + 1][1]; }
      }
      float us = 0.f;
#pragma unroll
      for (int x = 0; x < (WIDE ? 2 : 1); ++x) {
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) {                  // the four lanes of a head hold different keys
          const float m2 = __shfl_xor_sync(0xffffffffu, m[x], o), s2 = __shfl_xor_sync(0xffffffffu, ssum[x], o),
                      q2 = __shfl_xor_sync(0xffffffffu, sq[x], o);
          if (mode == PISA_SCORE_LSE) lse_merge(m[x], ssum[x], m2, s2);
          else { ssum[x] += s2; sq[x] += q2; }
        }
        if (parts == 1 && gid + 8 * x < NG) us += score_finish(mode, m[x], ssum[x], sq[x], C);
        if (PARTS == 2 && parts == 2 && gid + 8 * x < NG) {  // (max, sum) of this half to every CTA; tig takes every fourth one
          float* p = s_dyn + ((ci * 2 + pt) * NG + gid + 8 * x) * 2;
          for (int rk = tig; rk < CLU; rk += 4) {
            const uint32_t q = remote_smem(p, rk);
            st_remote(q, m[x]);
            st_remote(q + 4, ssum[x]);
          }
        }
      }
      __syncwarp();
      if (parts == 1) {
        us += __shfl_xor_sync(0xffffffffu, us, 4);
        us += __shfl_xor_sync(0xffffffffu, us, 8);
        us += __shfl_xor_sync(0xffffffffu, us, 16);
        if (lane < CLU) st_remote(remote_smem(&s_leaf[ci], lane), rankable(us));
      }
    }
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();

  // ---------------------------------------------------------------- 3. final Select_K (every CTA)
  if (PARTS == 2 && parts == 2 && tid >= 1 && tid <= n_sc) {
    const float* p = s_dyn + tid * 4 * NG;
    float us = 0.f;
#pragma unroll
    for (int hh = 0; hh < NG; ++hh) {
      float m = p[2 * hh], ssum = p[2 * hh + 1];
      lse_merge(m, ssum, p[2 * (NG + hh)], p[2 * (NG + hh) + 1]);
      us += m + __logf(ssum);
    }
    s_leaf[tid] = rankable(us);
  }
  const int nsel = block_select(s_leaf, nV, K, s_cnt, [&](int p, int s) { s_sel[p] = cand[s]; });
  if (rank == 0 && tid < K) a.idx[(long long)bh * K + tid] = (tid < nsel) ? s_sel[tid] : -1;

  // ---------------------------------------------------------------- 4. attention
  float o_acc[NG][DV];
#pragma unroll
  for (int hh = 0; hh < NG; ++hh)
#pragma unroll
    for (int j = 0; j < DV; ++j) o_acc[hh][j] = 0.f;
  // heads gid, gid + 8 (base 2).  The maxima start at a finite value: parts without keys (sum 0) or with nothing but logits of
  // -inf then merge with weight 0 and parts that hold a NaN with NaN, none of them a case of its own.
  constexpr float kFloor = -3.0e38f;
  float m_run[2] = {kFloor, kFloor}, l_run[2] = {0.f, 0.f};
  const float sl2 = geo.scale * kLog2e;
  const int ppb = C / KT;                                  // pieces per block
  for (int u = gw; u < nsel * ppb; u += CLU * kDecWarps) {
    const int slot = u / ppb, key0 = s_sel[slot] * C + (u - slot * ppb) * KT;
    if (key0 > pos) continue;                              // the piece lies in the future
    RowFrag<D> kr[KT / 8];
#pragma unroll
    for (int x = 0; x < KT / 8; ++x) {
      const int t = key0 + 8 * x + gid;
      kr[x].load(kbh + (long long)t * geo.ks[1], t <= pos, lane);
    }
    // the piece's value rows (this lane's DV columns of each), in flight during the softmax
    uint32_t vraw[KT][DV / 2];
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) {
      const int t = key0 + kk;
#pragma unroll
      for (int j = 0; j < DV / 2; ++j) vraw[kk][j] = 0u;
      if (t <= pos) {
        const __nv_bfloat16* vr = vbh + (long long)t * geo.vs[1] + lane * DV;
        if constexpr (DV == 4) {
          const uint2 y = *reinterpret_cast<const uint2*>(vr);
          vraw[kk][0] = y.x; vraw[kk][DV / 2 - 1] = y.y;
        } else {
          vraw[kk][0] = *reinterpret_cast<const uint32_t*>(vr);
        }
      }
    }
    float z[KT / 8][4];
#pragma unroll
    for (int x = 0; x < KT / 8; ++x) {
      heads_dot<D, WIDE>(qf, kr[x], z[x]);
#pragma unroll
      for (int y = 0; y < 4; ++y) z[x][y] = (key0 + 8 * x + 2 * tig + (y & 1) <= pos) ? z[x][y] * sl2 : -CUDART_INF_F;
    }
#pragma unroll
    for (int y = 0; y < (WIDE ? 2 : 1); ++y) {             // head gid + 8 * y: its keys are in the four lanes of the group
      float tm = -CUDART_INF_F;
#pragma unroll
      for (int x = 0; x < KT / 8; ++x) tm = fmaxf(tm, fmaxf(z[x][2 * y], z[x][2 * y + 1]));
      tm = fmaxf(tm, __shfl_xor_sync(0xffffffffu, tm, 1));
      tm = fmaxf(tm, __shfl_xor_sync(0xffffffffu, tm, 2));
      const float mn = fmaxf(m_run[y], tm);
      const float alpha = ex2_approx(m_run[y] - mn);
      float ps = 0.f;
#pragma unroll
      for (int x = 0; x < KT / 8; ++x) {
        const float p0 = ex2_approx(z[x][2 * y] - mn), p1 = ex2_approx(z[x][2 * y + 1] - mn);
        ps += p0 + p1;
        if (gid + 8 * y < NG) {
          s_p[warp][8 * x + 2 * tig][gid + 8 * y] = p0;
          s_p[warp][8 * x + 2 * tig + 1][gid + 8 * y] = p1;
        }
      }
      l_run[y] = l_run[y] * alpha + ps;                    // this lane's keys only: the four lanes are added at the end
      m_run[y] = mn;
      if (tig == 0 && gid + 8 * y < NG) s_alpha[warp][gid + 8 * y] = alpha;
    }
    __syncwarp();
#pragma unroll
    for (int hh = 0; hh < NG; ++hh) {
      const float al = s_alpha[warp][hh];
#pragma unroll
      for (int j = 0; j < DV; ++j) o_acc[hh][j] *= al;
    }
#pragma unroll
    for (int kk = 0; kk < KT; ++kk) {                      // rows after pos hold zeros and weight 0
      float vv[DV];
#pragma unroll
      for (int j = 0; j < DV / 2; ++j) {
        vv[2 * j] = __uint_as_float(vraw[kk][j] << 16);
        vv[2 * j + 1] = __uint_as_float(vraw[kk][j] & 0xFFFF0000u);
      }
#pragma unroll
      for (int hh = 0; hh < NG; ++hh) {
        const float p = s_p[warp][kk][hh];
#pragma unroll
        for (int j = 0; j < DV; ++j) o_acc[hh][j] = fmaf(p, vv[j], o_acc[hh][j]);
      }
    }
    __syncwarp();
  }
  // ---------------------------------------------------------------- 5. merge
  float* mine = s_dyn + warp * W;
#pragma unroll
  for (int hh = 0; hh < NG; ++hh)
#pragma unroll
    for (int j = 0; j < DV; ++j) mine[hh * D + lane * DV + j] = o_acc[hh][j];
#pragma unroll
  for (int y = 0; y < (WIDE ? 2 : 1); ++y) {
    float l = l_run[y];
    l += __shfl_xor_sync(0xffffffffu, l, 1);
    l += __shfl_xor_sync(0xffffffffu, l, 2);
    if (tig == 0 && gid + 8 * y < NG) { mine[NG * D + gid + 8 * y] = m_run[y]; mine[NG * D + NG + gid + 8 * y] = l; }
  }
  __syncthreads();
  float* cta = s_dyn + kDecWarps * W;
  for (int e = tid; e < NG * D + NG; e += kDecThreads) {
    const bool is_o = e < NG * D;
    const int hh = is_o ? e / D : e - NG * D;
    float mw[kDecWarps], M = kFloor;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w) { mw[w] = s_dyn[w * W + NG * D + hh]; M = fmaxf(M, mw[w]); }
    float acc = 0.f;
#pragma unroll
    for (int w = 0; w < kDecWarps; ++w)
      acc += s_dyn[w * W + (is_o ? e : NG * D + NG + hh)] * ex2_approx(mw[w] - M);
    if (is_o) cta[e] = acc;
    else { cta[NG * D + hh] = M; cta[NG * D + NG + hh] = acc; }
  }
  __syncwarp();
  cluster_arrive();
  cluster_wait();
  constexpr int SLICE = (NG * D + CLU - 1) / CLU;          // outputs each CTA of the cluster merges and writes
  for (int x = tid; x < SLICE; x += kDecThreads) {
    const int e = rank * SLICE + x;
    if (e >= NG * D) break;
    const int hh = e / D;
    float mr[CLU], lr[CLU], orr[CLU], M = kFloor;
#pragma unroll
    for (int r = 0; r < CLU; ++r) {
      const uint32_t p = remote_smem(cta, r);
      mr[r] = ld_remote(p + (NG * D + hh) * 4);
      lr[r] = ld_remote(p + (NG * D + NG + hh) * 4);
      orr[r] = ld_remote(p + e * 4);
    }
#pragma unroll
    for (int r = 0; r < CLU; ++r) M = fmaxf(M, mr[r]);
    float acc = 0.f, den = 0.f;
#pragma unroll
    for (int r = 0; r < CLU; ++r)
    {
      const float f = ex2_approx(mr[r] - M);
      acc += orr[r] * f;
      den += lr[r] * f;
    }
    a.out[((long long)b * geo.Hq + (long long)h * NG + hh) * D + (e - hh * D)] = __float2bfloat16_rn(acc / den);
    if (e - hh * D == 0) a.lse[(long long)b * geo.Hq + (long long)h * NG + hh] = (M + log2f(den)) * kLn2;
  }
  __syncwarp();
  cluster_arrive();                                        // nobody leaves while its partial is still being read
  cluster_wait();
}

template <int D, int NG>
constexpr size_t decode_smem() { return (size_t)(kDecWarps + 1) * (NG * D + 2 * NG) * sizeof(float); }
// keys per attention piece: 32 where a thread has the registers to keep their rows in flight
constexpr int decode_piece(int NG, int MINB) { return (MINB == 1 && NG <= 8) ? 32 : 16; }
// clusters that refresh the pyramid, a warp per (batch, KV head)
inline int refresh_clusters(long long units, int clu) { return (int)((units + kDecWarps * clu - 1) / (kDecWarps * clu)); }

template <int D, int NG, int MINB, int CLU, bool MOM>
int launch_decode(const Geometry& g, const DecArgs& a, cudaStream_t s) {
  constexpr auto kern = decode_step_kernel<D, NG, decode_piece(NG, MINB), MINB, CLU, MOM>;
  if (CLU > 8) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) { record_cuda_error("decode_step attr", e); return PISA_ERR_CUDA; }
  }
  int refresh = refresh_clusters(a.units, CLU);
  if (a.units + refresh > 65535) {                         // more clusters than a grid's y holds
    refresh = 0;
    const int st = launch_dependent<decode_refresh_kernel<D>>("decode_refresh", dim3((unsigned)((a.units + kDecWarps - 1) / kDecWarps)),
                                                              kDecThreads, 0, s, g, a);
    if (st != PISA_OK) return st;
  }
  return launch_dependent<kern>("decode_step", dim3(CLU, (unsigned)(a.units + refresh)), kDecThreads, decode_smem<D, NG>(), s, g, a);
}
// How many clusters of this instantiation the GPU holds at once (clusters are placed inside one GPC, so
// this is less than SMs * MINB / CLU); asked of the driver once per instantiation and device, again if it could not say.
template <int D, int NG, int CLU>
int resident_clusters() {
  constexpr int kMaxDev = 64;
  static std::atomic<int> cached[kMaxDev] = {};           // clusters + 1
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return 0; }
  const bool keep = dev >= 0 && dev < kMaxDev;
  const int known = keep ? cached[dev].load(std::memory_order_relaxed) : 0;
  if (known > 0) return known - 1;
  const size_t smem = decode_smem<D, NG>();
  constexpr auto kern = decode_step_kernel<D, NG, decode_piece(NG, 1), 1, CLU, false>;
  allow_smem<kern>(smem);
  if (CLU > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(CLU, 1024);
  cfg.blockDim = dim3(kDecThreads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CLU; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  if (keep) cached[dev].store(n + 1, std::memory_order_relaxed);
  return n;
}

// The widest cluster whose clusters (the refreshing ones included) are all resident at once at one CTA per SM (all
// registers); beyond that clusters of two at two CTAs per SM, in waves once even those do not fit.  The moment scores take
// the two ends only.
template <int D, int NG>
int launch_decode_heads(const Geometry& g, const DecArgs& a, cudaStream_t s) {
  auto fits = [&](int clu, int resident) { return a.units + refresh_clusters(a.units, clu) <= resident; };
  if (g.score_mode != PISA_SCORE_LSE)
    return fits(8, resident_clusters<D, NG, 8>()) ? launch_decode<D, NG, 1, 8, true>(g, a, s) : launch_decode<D, NG, 2, 2, true>(g, a, s);
  if (fits(16, resident_clusters<D, NG, 16>())) return launch_decode<D, NG, 1, 16, false>(g, a, s);
  if (fits(8, resident_clusters<D, NG, 8>())) return launch_decode<D, NG, 1, 8, false>(g, a, s);
  if (fits(4, resident_clusters<D, NG, 4>())) return launch_decode<D, NG, 1, 4, false>(g, a, s);
  if (fits(2, resident_clusters<D, NG, 2>())) return launch_decode<D, NG, 1, 2, false>(g, a, s);
  return launch_decode<D, NG, 2, 2, false>(g, a, s);
}
template <int D>
int launch_decode_dim(const Geometry& g, const DecArgs& a, cudaStream_t s) {
  switch (g.G) {
    case 1: return launch_decode_heads<D, 1>(g, a, s);
    case 2: return launch_decode_heads<D, 2>(g, a, s);
    case 4: return launch_decode_heads<D, 4>(g, a, s);
    case 8: return launch_decode_heads<D, 8>(g, a, s);
    case 16: return launch_decode_heads<D, 16>(g, a, s);
    default: return PISA_ERR_UNSUPPORTED;
  }
}

}  // namespace

int launch_decode_d64(const Geometry& g, const DecArgs& a, cudaStream_t s);
int launch_decode_d128(const Geometry& g, const DecArgs& a, cudaStream_t s);

}  // namespace pisa
