// Select_K with one THREAD per (b, KV head, token) (see query_major.cuh; Sec. 3.2 "Coarse-to-fine block selection").
//
// A warp that selects for one token spends its instructions on shuffles: 21 exchange steps of two shuffles each for 64
// candidates, 32 lanes wide, per token and level.  Here a lane owns a token, holds its candidates' scores in registers
// and runs a whole odd-even merge sort on them: 543 comparators of two instructions for 64 candidates, i.e. 34 issue
// slots per token instead of about 250.  The scores of the levels above the leaves come from the table the dense scoring
// wrote, those of the leaves from its leaf table (FULL) or from the list-driven scoring (FINAL).
#pragma once

#include <math_constants.h>

#include "launch.cuh"
#include "pisa_tensor.cuh"
#include "query_major.cuh"

namespace pisa {

namespace {

constexpr int kSelThreads = 64;

// FULL: top level .. leaves.  STAGE1: top level .. 2, kept level-2 nodes out.  FINAL: leaves only, kept level-2 nodes in.
enum { kSelFull = 0, kSelStage1 = 1, kSelFinal = 2 };

struct SelArgs {
  int32_t* par;            // STAGE1: out, FINAL: in   [B, Hkv, N, K]
  const float* blk;        // FINAL: leaf scores per candidate, [B, Hkv, N, g*K, G]
  int32_t* idx;            // [Hkv, len, K] per sequence
  float* margin;           // null or [B, Hkv, N] (uniform batches)
  float* lse;              // null or [Hq, len] per sequence
  float* sel_lse;          // null or [B, Hq, N, K] (uniform batches)
  int vec;                 // rows of par / idx can be written four entries at a time
};

__device__ __forceinline__ void cmp_desc(float& a, float& b) {
  const float hi = fmaxf(a, b), lo = fminf(a, b);
  a = hi; b = lo;
}
// Batcher's odd-even merge sort (K. E. Batcher, 1968), descending, fully unrolled on registers
template <int NC, int LO, int N, int R>
__device__ __forceinline__ void oe_merge(float (&v)[NC]) {
  constexpr int M = R * 2;
  if constexpr (M < N) {
    oe_merge<NC, LO, N, M>(v);
    oe_merge<NC, LO + R, N, M>(v);
#pragma unroll
    for (int i = LO + R; i + R < LO + N; i += M) cmp_desc(v[i], v[i + R]);
  } else {
    cmp_desc(v[LO], v[LO + R]);
  }
}
template <int NC, int LO, int N>
__device__ __forceinline__ void oe_sort(float (&v)[NC]) {
  if constexpr (N > 1) {
    oe_sort<NC, LO, N / 2>(v);
    oe_sort<NC, LO + N / 2, N / 2>(v);
    oe_merge<NC, LO, N, 1>(v);
  }
}

template <int G>   // G consecutive floats, as wide as their alignment allows
__device__ __forceinline__ void load_heads(const float* p, float (&x)[G]) {
  if constexpr (G == 1) x[0] = p[0];
  else if constexpr (G == 2) { const float2 y = *reinterpret_cast<const float2*>(p); x[0] = y.x; x[1] = y.y; }
  else {
#pragma unroll
    for (int i = 0; i < G; i += 4) {
      const float4 y = *reinterpret_cast<const float4*>(p + i);
      x[i] = y.x; x[i + 1] = y.y; x[i + 2] = y.z; x[i + 3] = y.w;
    }
  }
}
template <int G>
__device__ __forceinline__ float sum_heads(const float* p) {
  float x[G];
  load_heads<G>(p, x);
  if constexpr (G == 4) return (x[0] + x[1]) + (x[2] + x[3]);
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < G; ++i) s += x[i];
  return s;
}

// Select_K among nV > K scores by counting, a NaN last (the sorting network's results assume an order)
struct Ranked { uint4 keep; float cut, next; };                   // one bit per candidate; the K-th largest score and the one after
__device__ __noinline__ Ranked select_by_rank(const float* u, int nV, int K) {
  Ranked r;
  r.keep = make_uint4(0u, 0u, 0u, 0u);
  for (int i = 0; i < nV; ++i) {
    const float ui = rankable(u[i * kSelThreads]);
    int rank = 0;
    for (int j = 0; j < nV; ++j) {
      const float uj = rankable(u[j * kSelThreads]);
      rank += uj > ui || (uj == ui && j < i);
    }
    const uint32_t bit = rank < K ? 1u << (i & 31) : 0u;
    if (i < 32) r.keep.x |= bit;
    else if (i < 64) r.keep.y |= bit;
    else if (i < 96) r.keep.z |= bit;
    else r.keep.w |= bit;
    if (rank == K - 1) r.cut = ui;
    if (rank == K) r.next = ui;
  }
  return r;
}

// NC: candidates a token can have at a level (g * K rounded up), FAN = g.
// Bound by the latency of its loads, twelve warps per SM waiting; bounding the registers for more (10, 12, 14 CTAs per SM)
// spills the sorting network: 575 us -> 576, 595, 600 for a forward of 8192 tokens, 16 heads.
template <int NC, int FAN, int G, int MODE>
__global__ void __launch_bounds__(kSelThreads) qm_select_kernel(Geometry geo, qm::Args a, SelArgs sa) {
  extern __shared__ float s_mem[];
  constexpr int LGF = (FAN == 2) ? 1 : 2, NW = (NC + 31) / 32;
  const int tid = threadIdx.x, K = geo.K;
  float* s_u = s_mem + tid;                                       // [NC][threads] scores of the level, candidate order
  int* s_kept = reinterpret_cast<int*>(s_mem + NC * kSelThreads) + tid;   // [2][K][threads] kept nodes, ping-pong
  grid_dependency();
  if (a.ctr != nullptr && blockIdx.x == 0 && blockIdx.y == 0 && tid == 0) *a.ctr = 0;
  const int lgC = a.lgC, h = blockIdx.y;
  long long r = (long long)blockIdx.x * kSelThreads + tid;
  qm::Seq q;
  int t;
  if (a.seqs == nullptr) {
    const int rows = a.t1 - a.t0;
    const int b = (int)(r / rows);
    if (b >= geo.B) return;
    t = a.t0 + (int)(r - (long long)b * rows);
    q = qm::uniform_seq(geo, a, b, 0);
  } else {
    int lo = 0, hi = a.nseq;                                      // sequences in order of their first token
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (a.seqs[mid].row0 <= r) lo = mid; else hi = mid;
    }
    q = a.seqs[lo];
    t = (int)(r - q.row0);
    if (t >= q.len) return;
  }
  const int len = q.len, c = t >> lgC;
  const int M1 = qm::level_nodes(len, lgC, LGF, 1);
  const int top = qm::top_level(len, lgC, LGF, K);
  const int width = qm::table_width(len, lgC, LGF, top);
  const long long row = (long long)h * len + t;                   // row of the sequence's tables and outputs
  const long long urow = (a.seqs == nullptr)                      // row of a uniform batch
                             ? ((long long)q.batch * geo.Hkv + h) * geo.N + t : row;
  const float* up = a.up + q.up_off +
                    (a.seqs ? row : ((long long)(q.batch * geo.Hkv + h) * (a.t1 - a.t0) + (t - a.t0))) * width;
  const float* leaves = (MODE == kSelFinal) ? sa.blk + urow * ((long long)K << LGF) * G
                                            : a.leaf + q.leaf_off + row * (long long)qm::level_width(M1) * G;

  int buf = 0, nk = 0;
  float gap = CUDART_INF_F;
  int l0;                                                          // level the walk starts at
  bool first = true;                                               // its candidates are simply the nodes 0 .. anc(c)
  if (MODE == kSelFinal) {
    l0 = 1;
    first = false;
    const int32_t* pr = sa.par + urow * K;
    for (int s = 0; s < K; ++s) {
      int p = pr[s];
      if ((geo.debug & PISA_DEBUG_BOUNDS) && p != -1 && !bounds_ok(p, qm::level_nodes(len, lgC, LGF, 2), a.status)) p = -1;
      if (p < 0) break;
      s_kept[s * kSelThreads] = p;
      nk = s + 1;
    }
    if (sa.margin != nullptr) gap = sa.margin[urow];
  } else {
    l0 = max(top, MODE == kSelStage1 ? 2 : 1);
  }
  int off = 0;                                                     // column of level l in the node table
  for (int l = 2; l < l0; ++l) off += qm::level_width(qm::level_nodes(len, lgC, LGF, l));
  for (int l = l0; l >= (MODE == kSelStage1 ? 2 : 1); --l) {
    const int sh = qm::level_shift(lgC, LGF, l);
    const int anc = t >> sh;
    const int fp = (c >= 1) ? (((c - 1) << lgC) >> sh) : 0;        // ancestor of the previous leaf
    int* kin = s_kept + buf * K * kSelThreads;
    int* kout = s_kept + (buf ^ 1) * K * kSelThreads;
    const int n = first ? anc + 1 : nk << LGF;
    // candidates that do not start after the query's leaf form a prefix of nV; the kept nodes always include the
    // ancestors of the first, the previous and the current leaf, so these are candidate 0 and the last one or two
    int nV = n;
    if (!first && nk > 0) nV = n - max(0, (kin[(nk - 1) * kSelThreads] << LGF) + FAN - 1 - anc);
    const int nEnd = nV - 1 - (fp != anc);                         // scored: candidates 1 .. nEnd - 1
    uint32_t keep[NW];
    if (nV > K) {
      float v[NC];
#pragma unroll
      for (int p = 0; p < NC / FAN; ++p) {
        float x[FAN];
#pragma unroll
        for (int j = 0; j < FAN; ++j) x[j] = 0.f;
        if (p * FAN < nEnd) {
          const int node0 = (first ? p : kin[p * kSelThreads]) << LGF;
          if (MODE != kSelStage1 && l == 1) {
            const float* src = leaves + (long long)((MODE == kSelFinal) ? p * FAN : node0) * G;
            if constexpr (G == 1) {
              load_heads<FAN>(src, x);
            } else {
#pragma unroll
              for (int j = 0; j < FAN; ++j) x[j] = sum_heads<G>(src + j * G);
            }
          } else if (MODE != kSelFinal) {
            load_heads<FAN>(up + off + node0, x);
          }
        }
#pragma unroll
        for (int j = 0; j < FAN; ++j) {
          const int i = p * FAN + j;
          const float sc = (i >= nV) ? -CUDART_INF_F : (i == 0 || i >= nEnd) ? forced_score(i) : x[j];
          v[i] = sc;
          s_u[i * kSelThreads] = sc;
        }
      }
      oe_sort<NC, 0, NC>(v);
      float T = 0.f;                                               // K-th largest
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (i == K - 1) T = v[i];
      float T1 = 0.f;                                              // and the next one
      if (sa.margin != nullptr) {
#pragma unroll
        for (int i = 0; i < NC; ++i)
          if (i == K) T1 = v[i];
      }
      int cnt = 0;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        uint32_t m = 0u;
#pragma unroll
        for (int i = w * 32; i < min(NC, w * 32 + 32); ++i) m |= (s_u[i * kSelThreads] >= T) ? (1u << (i & 31)) : 0u;
        const int valid = nV - w * 32;
        keep[w] = (valid >= 32) ? m : (valid > 0 ? m & ((1u << valid) - 1u) : 0u);
        cnt += __popc(keep[w]);
      }
      int room = K;                                                // less the candidates above the cut
      if (cnt > K) {                                               // equal scores at the cut: the smaller positions stay
        for (int w = 0; w < NW; ++w)
          for (uint32_t m = keep[w]; m != 0u; m &= m - 1u) room -= s_u[(w * 32 + __ffs(m) - 1) * kSelThreads] > T;
        int eq = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w)
          for (uint32_t m = keep[w]; m != 0u; m &= m - 1u) {
            const int i = __ffs(m) - 1;
            if (s_u[(w * 32 + i) * kSelThreads] == T && ++eq > room) keep[w] &= ~(1u << i);
          }
      }
      // T is the K-th largest exactly if at least K candidates reach it and fewer than K exceed it.  A comparator replaces a
      // NaN by a copy of its other input, so with scores that are not numbers it may be another one: then by rank, NaN last
      // (clamping every score instead costs 3 us of the 530 of a forward of 8192 tokens, 16 heads)
      if (cnt < K || room < 1) {
        const Ranked r = select_by_rank(s_u, nV, K);
        T = r.cut;
        T1 = r.next;
#pragma unroll
        for (int w = 0; w < NW; ++w) keep[w] = w == 0 ? r.keep.x : w == 1 ? r.keep.y : w == 2 ? r.keep.z : r.keep.w;
      }
      if (sa.margin != nullptr && T < kForcedFloor) gap = fminf(gap, (T - T1) / fmaxf(fabsf(T), 1.f));
    } else {
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const int valid = nV - w * 32;
        keep[w] = (valid >= 32) ? 0xffffffffu : (valid > 0 ? (1u << valid) - 1u : 0u);
      }
    }
    int kept = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w)
      for (uint32_t m = keep[w]; m != 0u && kept < K; m &= m - 1u) {
        const int i = w * 32 + __ffs(m) - 1;
        kout[kept * kSelThreads] = first ? i : (kin[(i >> LGF) * kSelThreads] << LGF) + (i & (FAN - 1));
        if (MODE == kSelFinal) reinterpret_cast<int*>(s_u)[kept * kSelThreads] = i;      // where its scores are
        ++kept;
      }
    nk = kept;
    buf ^= 1;
    first = false;
    if (l > 2) off -= qm::level_width(qm::level_nodes(len, lgC, LGF, l - 1));
  }
  const int* kf = s_kept + buf * K * kSelThreads;
  int32_t* dst = (MODE == kSelStage1) ? sa.par + urow * K : sa.idx + geo.Hkv * K * q.cu + row * K;
  if (sa.vec) {
    for (int s = 0; s < K; s += 4) {
      int4 o;
      o.x = (s < nk) ? kf[s * kSelThreads] : -1;
      o.y = (s + 1 < nk) ? kf[(s + 1) * kSelThreads] : -1;
      o.z = (s + 2 < nk) ? kf[(s + 2) * kSelThreads] : -1;
      o.w = (s + 3 < nk) ? kf[(s + 3) * kSelThreads] : -1;
      *reinterpret_cast<int4*>(dst + s) = o;
    }
  } else {
    for (int s = 0; s < K; ++s) dst[s] = (s < nk) ? kf[s * kSelThreads] : -1;
  }
  if (sa.margin != nullptr) sa.margin[urow] = gap;
  if (MODE == kSelStage1) return;
  auto leaf_at = [&](int s) {
    const int i = (MODE == kSelFinal) ? reinterpret_cast<int*>(s_u)[s * kSelThreads] : kf[s * kSelThreads];
    return leaves + (long long)i * G;
  };
  if (sa.lse != nullptr) {
    float m[G], ssum[G];
#pragma unroll
    for (int hh = 0; hh < G; ++hh) { m[hh] = -CUDART_INF_F; ssum[hh] = 0.f; }
    constexpr int U = G <= 4 ? 8 : 2;                              // leaves in flight
    for (int s0 = 0; s0 < nk; s0 += U) {
      float x[U][G];
#pragma unroll
      for (int u = 0; u < U; ++u) load_heads<G>(leaf_at(min(s0 + u, nk - 1)), x[u]);
#pragma unroll
      for (int hh = 0; hh < G; ++hh) {
        float mn = m[hh];
#pragma unroll
        for (int u = 0; u < U; ++u) mn = fmaxf(mn, x[u][hh]);
        float sum = ssum[hh] != 0.f ? ssum[hh] * __expf(m[hh] - mn) : 0.f;     // (0: nothing yet, m = -inf)
#pragma unroll
        for (int u = 0; u < U; ++u) sum += s0 + u < nk ? __expf(x[u][hh] - mn) : 0.f;
        m[hh] = mn;
        ssum[hh] = sum;
      }
    }
#pragma unroll
    for (int hh = 0; hh < G; ++hh) sa.lse[(long long)geo.Hq * q.cu + (long long)(h * G + hh) * len + t] = m[hh] + __logf(ssum[hh]);
  }
  if (sa.sel_lse != nullptr)
    for (int s = 0; s < K; ++s)
#pragma unroll
      for (int hh = 0; hh < G; ++hh)
        sa.sel_lse[(((long long)q.batch * geo.Hq + h * G + hh) * geo.N + t) * K + s] =
            (s < nk) ? leaf_at(s)[hh] : -CUDART_INF_F;
  if (a.bits != nullptr) {
    const int W = (M1 + 31) >> 5;
    uint32_t* bw = a.bits + q.bits_off + row * W;
    int s = 0;
    for (int w = 0; w < W; ++w) {
      uint32_t word = 0u;
      for (; s < nk && (kf[s * kSelThreads] >> 5) == w; ++s) word |= 1u << (kf[s * kSelThreads] & 31);
      bw[w] = word;
    }
  }
}

template <int NC, int FAN, int G, int MODE>
int launch_sel(const Geometry& g, const qm::Args& a, const SelArgs& sa, long long rows, cudaStream_t s) {
  const size_t smem = (size_t)kSelThreads * (NC + 2 * g.K) * 4;
  dim3 grid((unsigned)((rows + kSelThreads - 1) / kSelThreads), (unsigned)g.Hkv);
  return launch_dependent<qm_select_kernel<NC, FAN, G, MODE>>("qm_select", grid, kSelThreads, smem, s, g, a, sa);
}
template <int NC, int FAN, int MODE>
int launch_sel_g(const Geometry& g, const qm::Args& a, const SelArgs& sa, long long rows, cudaStream_t s) {
  if constexpr (MODE == kSelStage1) return launch_sel<NC, FAN, 1, MODE>(g, a, sa, rows, s);
  else
    switch (g.G) {
      case 1: return launch_sel<NC, FAN, 1, MODE>(g, a, sa, rows, s);
      case 2: return launch_sel<NC, FAN, 2, MODE>(g, a, sa, rows, s);
      case 4: return launch_sel<NC, FAN, 4, MODE>(g, a, sa, rows, s);
      case 8: return launch_sel<NC, FAN, 8, MODE>(g, a, sa, rows, s);
      case 16: return launch_sel<NC, FAN, 16, MODE>(g, a, sa, rows, s);
      default: return PISA_ERR_UNSUPPORTED;
    }
}
// rows: tokens of all sequences (uniform: B * (t1 - t0))
template <int MODE>
int launch_sel_mode(const Geometry& g, const qm::Args& a, SelArgs sa, long long rows, cudaStream_t s) {
  const int gK = g.g * g.K;
  const void* rows_out = (MODE == kSelStage1) ? (const void*)sa.par : (const void*)sa.idx;
  sa.vec = (g.K & 3) == 0 && (reinterpret_cast<uintptr_t>(rows_out) & 15u) == 0;
  if (g.g == 2) {
    if (gK <= 16) return launch_sel_g<16, 2, MODE>(g, a, sa, rows, s);
    if (gK <= 32) return launch_sel_g<32, 2, MODE>(g, a, sa, rows, s);
    return launch_sel_g<64, 2, MODE>(g, a, sa, rows, s);               // K <= 32
  }
  if (gK <= 16) return launch_sel_g<16, 4, MODE>(g, a, sa, rows, s);
  if (gK <= 32) return launch_sel_g<32, 4, MODE>(g, a, sa, rows, s);
  if (gK <= 64) return launch_sel_g<64, 4, MODE>(g, a, sa, rows, s);
  return launch_sel_g<128, 4, MODE>(g, a, sa, rows, s);
}

}  // namespace
}  // namespace pisa
