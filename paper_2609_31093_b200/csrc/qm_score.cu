// Dense scoring of leaves and upper-level nodes, query-major (see query_major.cuh).
//
// A work item is NT 128-row tiles of one KV head (consecutive token ranges), one CTA each.  Roles: warp 0 TMA producer,
// warp 1 UMMA issuer, from warp 4 on groups of four epilogue warps (TMEM lane quarter = warp % 4), one group per (tile,
// step parity).  A step is 128 rows of the B operand: keys of one or two leaves, or 128 consecutive rows of a pyramid
// level (the children of 128 / g nodes of the level above).
// What bounds it: per step and tile 1024 cycles of exponentials (one per row and key, 16 per clock), 512 of the tensor
// pipe -- and the 32 KB (d = 128) of keys from L2, which an SM takes in at about 22 bytes per clock.  One tile per load
// (two CTAs per SM) ran at that rate, 1470 cycles per tile and step with the epilogue switched off; two tiles share a
// load, one CTA of 20 warps per SM.  Short batches, whose pairs of tiles would not fill the SMs, keep one tile per CTA.
#include "launch.cuh"
#include "lse_chunk.cuh"
#include "pisa_tensor.cuh"
#include "query_major.cuh"
#include "tc_utils.cuh"
#include "tma_map.cuh"

namespace pisa {

using namespace tc;

namespace {

constexpr int kMaxUpSteps = 64;
// of every eight pairs of exponentials, how many take the FMA pipe: with none the special-function unit is busy 75 % of the
// time.  8192 tokens, 4 x 16 heads, G = 4: none 734 us, one 708, two 697, three 724, four 782; C = 128, 32 heads: 353, 335,
// 326, 343, 368.  (The attention kernel, which waits for the latency of its softmax, gets slower with any of them.)
constexpr int kPoly = 2;

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// group-summed natural scores of the 32 / FAN nodes whose children are these 32 columns.  The sum over the G lanes of a
// token is a reduce-scatter (half of the live values per step: 12 shuffles for sixteen nodes and G = 4, 15 for G = 16,
// where adding all of them in every lane takes 32 and 64), which leaves each lane the nodes it stores.
template <int FAN, int G>
__device__ __forceinline__ void score_nodes(const uint32_t (&r)[32], float sl2, int head, float* dst, int node0, int width, bool live) {
  constexpr int NN = 32 / FAN, KEEP = NN / G > 0 ? NN / G : 1;
  float u[NN];
#pragma unroll
  for (int i = 0; i < NN; ++i) {
    if (FAN == 2) {
      const float za = __uint_as_float(r[2 * i]) * sl2, zb = __uint_as_float(r[2 * i + 1]) * sl2;
      u[i] = fmaxf(za, zb) + lg2_approx(1.f + ex2_approx(-fabsf(za - zb)));
    } else {
      float m = __uint_as_float(r[FAN * i]);
#pragma unroll
      for (int j = 1; j < FAN; ++j) m = fmaxf(m, __uint_as_float(r[FAN * i + j]));
      m *= sl2;
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < FAN; ++j) s += ex2_approx(fmaf(__uint_as_float(r[FAN * i + j]), sl2, -m));
      u[i] = m + lg2_approx(s);
    }
  }
  int base = 0;                                                  // first node this lane keeps
#pragma unroll
  for (int o = 1, cnt = NN; o < G; o <<= 1) {
    if (cnt > 1) {
      const bool up = (head & o) != 0;
      cnt >>= 1;
#pragma unroll
      for (int i = 0; i < NN / 2; ++i)
        if (i < cnt) {
          const float send = up ? u[i] : u[i + cnt], mine = up ? u[i + cnt] : u[i];
          u[i] = mine + __shfl_xor_sync(0xffffffffu, send, o);
        }
      base += up ? cnt : 0;
    } else {
      u[0] += __shfl_xor_sync(0xffffffffu, u[0], o);
    }
  }
  if (!live || (G > NN && head >= NN)) return;
  float* p = dst + node0 + base;
  if constexpr (KEEP >= 4) {
#pragma unroll
    for (int i = 0; i < KEEP; i += 4)
      if (node0 + base + i < width)
        *reinterpret_cast<float4*>(p + i) = make_float4(u[i] * kLn2, u[i + 1] * kLn2, u[i + 2] * kLn2, u[i + 3] * kLn2);
  } else if (node0 + base < width) {
#pragma unroll
    for (int i = 0; i < KEEP; ++i) p[i] = u[i] * kLn2;
  }
}
template <int FAN>
__device__ __forceinline__ void score_nodes_g(const uint32_t (&r)[32], float sl2, int G, int head, float* dst, int node0, int width,
                                              bool live) {
  switch (G) {
    case 1: score_nodes<FAN, 1>(r, sl2, head, dst, node0, width, live); break;
    case 2: score_nodes<FAN, 2>(r, sl2, head, dst, node0, width, live); break;
    case 4: score_nodes<FAN, 4>(r, sl2, head, dst, node0, width, live); break;
    case 8: score_nodes<FAN, 8>(r, sl2, head, dst, node0, width, live); break;
    default: score_nodes<FAN, 16>(r, sl2, head, dst, node0, width, live); break;
  }
}

// stages of the key ring: two CTAs per SM with one tile each, one CTA with two
__host__ __device__ constexpr int score_stages(int D, int NT) { return (D == 128 && NT == 1) ? 2 : 4; }

template <int D, int C, int NT>
__global__ void __launch_bounds__(128 + 256 * NT, 3 - NT)
qm_score_kernel(Geometry geo, qm::Args a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                const __grid_constant__ CUtensorMap tm_p) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = D / 64, SLAB = 128 * 128, STAGE = KS * SLAB, NK = score_stages(D, NT);
  constexpr uint32_t TM_COLS = 256 * NT;       // two accumulators of 128 columns per tile
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;
  uint8_t* sK = smem + NT * STAGE;
  __shared__ uint64_t q_full, k_full[NK], k_empty[NK], t_full[2 * NT], t_empty[2 * NT];
  __shared__ int4 s_up[kMaxUpSteps];           // upper-level steps: (pyramid row of the first child, first node, column, width)
  __shared__ int s_nup;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int lgC = a.lgC, lgg = a.lgg, lgG = a.lgG, tpt = 128 >> lgG, G = geo.G;
  grid_dependency();
  const qm::Tile tl = qm::locate(geo, a, blockIdx.x, NT);
  const int len = tl.q.len, h = tl.h, tile0 = tl.tile * tpt * NT;
  const int t_last = min(len, tile0 + NT * tpt) - 1;
  const int n_leaf = a.want_leaf ? (t_last >> 7) + 1 : 0;
  const int top = qm::top_level(len, lgC, lgg, geo.K);
  const int width = qm::table_width(len, lgC, lgg, top);

  if (tid == 0) {
    mbar_init(&q_full, 1);
    for (int i = 0; i < NK; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1); }
    for (int i = 0; i < 2 * NT; ++i) { mbar_init(&t_full[i], 1); mbar_init(&t_empty[i], 4); }
    s_fail = 0;
    mbar_fence_init();
    // children of the level-l nodes 0 .. anc(t_last) - 1 (the last node is forced, never scored), where a row can prune
    int n = 0, col = 0, row0 = tl.q.pyr_row;
    for (int l = 2; l <= top; ++l) {
      const int Mb = qm::level_nodes(len, lgC, lgg, l - 1), Ml = qm::level_nodes(len, lgC, lgg, l);
      const int anc = t_last >> qm::level_shift(lgC, lgg, l);
      const int base = a.seqs ? row0 + h * Mb
                              : (int)(geo.level_off[l - 1] / D) + (tl.q.batch * geo.Hkv + h) * Mb;
      if (anc + 1 > geo.K)
        for (int r = 0; r < (anc << lgg) && n < kMaxUpSteps; r += 128, ++n)
          s_up[n] = make_int4(base + r, r >> lgg, col, qm::level_width(Ml));
      col += qm::level_width(Ml);
      row0 += geo.Hkv * Mb;
    }
    s_nup = n;
  }
  if (warp == 0) { tmem_alloc(&tmem_slot, TM_COLS); tmem_relinquish(); }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  const int n_steps = n_leaf + s_nup;

  if (warp == 0) {
    if (lane == 0 && n_steps > 0) {
      mbar_arrive_expect_tx(&q_full, (uint32_t)(NT * STAGE));
      for (int x = 0; x < NT; ++x)
        for (int ks = 0; ks < KS; ++ks)
          tma_load_4d(smem_u32(sQ + x * STAGE + ks * SLAB), &tm_q, &q_full, ks * 64, h * G, tl.q.tok + tile0 + x * tpt, tl.q.batch);
      for (int i = 0; i < n_steps; ++i) {
        const int s = i % NK;
        if (i >= NK && !mbar_wait_bounded(&k_empty[s], (uint32_t)((i / NK - 1) & 1))) { s_fail = 1; break; }
        mbar_arrive_expect_tx(&k_full[s], (uint32_t)STAGE);
        for (int ks = 0; ks < KS; ++ks) {
          const uint32_t dst = smem_u32(sK + s * STAGE + ks * SLAB);
          if (i < n_leaf) tma_load_4d(dst, &tm_k, &k_full[s], ks * 64, h, tl.q.tok + i * 128, tl.q.batch);
          else tma_load_3d(dst, &tm_p, &k_full[s], ks * 64, s_up[i - n_leaf].x, 0);
        }
      }
    }
  } else if (warp == 1) {
    const uint32_t idesc = make_idesc_bf16(128, 128, 0, 0);
    bool ok = n_steps == 0 || mbar_wait_bounded(&q_full, 0u);
    for (int i = 0; i < n_steps && ok; ++i) {
      const int s = i % NK, par = i & 1;
      ok = mbar_wait_bounded(&k_full[s], (uint32_t)((i / NK) & 1));
#pragma unroll 1
      for (int x = 0; x < NT && ok; ++x) {
        const int buf = x * 2 + par;
        if (i >= 2) ok = mbar_wait_bounded(&t_empty[buf], (uint32_t)(((i >> 1) - 1) & 1));
        ok = __all_sync(0xffffffffu, ok && !s_fail);
        if (!ok) break;
        tcgen05_fence_after_sync();
        const uint32_t q0 = desc_lo(smem_u32(sQ) + (uint32_t)(x * STAGE), 0), k0 = desc_lo(smem_u32(sK) + (uint32_t)(s * STAGE), 0);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk) {
            const uint32_t o = (uint32_t)((kk >> 2) * SLAB + (kk & 3) * 32) >> 4;
            umma_bf16(tmem + (uint32_t)(buf * 128), desc64(q0 + o), desc64(k0 + o), idesc, kk > 0);
          }
          if (x == NT - 1) umma_commit(&k_empty[s]);
          umma_commit(&t_full[buf]);
        }
        __syncwarp();
      }
    }
    if (!ok) s_fail = 1;
  } else if (warp >= 4) {
    const int grp = (warp - 4) >> 2, quarter = warp & 3;       // group = tile * 2 + step parity
    const int row = quarter * 32 + lane, head = row & (G - 1);
    const int t = tile0 + (grp >> 1) * tpt + (row >> lgG);
    const bool live = t < len;
    const int c = t >> lgC, M1 = (len + C - 1) >> lgC;
    const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(grp * 128);
    const float sl2 = geo.scale * kLog2e;
    float* leaf_row = a.leaf + tl.q.leaf_off + (((long long)h * len + t) * qm::level_width(M1)) * G + head;
    float* up_row = a.up + tl.q.up_off +
                    (a.seqs ? ((long long)h * len + t)
                            : ((long long)(tl.q.batch * geo.Hkv + h) * (a.t1 - a.t0) + (t - a.t0))) * width;
    for (int i = grp & 1; i < n_steps; i += 2) {
      if (!mbar_wait_bounded(&t_full[grp], (uint32_t)((i >> 1) & 1)) || s_fail) { s_fail = 1; break; }
      tcgen05_fence_after_sync();
      auto handed_back = [&]() {                                // the accumulator is in registers
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&t_empty[grp]);
      };
      if (i < n_leaf) {
#pragma unroll
        for (int r = 0; r < 128 / C; ++r) {
          const int leaf = i * (128 / C) + r;
          // causally visible keys of this leaf for this row: all of an earlier leaf, keys <= t of the row's own
          const int ncols = !live ? 0 : (leaf < c ? C : (leaf == c ? t - (leaf << lgC) + 1 : 0));
          float m = -CUDART_INF_F, ssum = 0.f;
          const bool any = __any_sync(0xffffffffu, ncols > 0);
#pragma unroll
          for (int q = 0; q < C / 32; ++q) {
            uint32_t rr[32];
            if (any) {
              tmem_ld_32x32(base + (uint32_t)(r * C + q * 32), rr);
              tmem_ld_wait();
            }
            if (r == 128 / C - 1 && q == C / 32 - 1) handed_back();
            if (any) {
              const int nv = max(0, min(32, ncols - 32 * q));
              if (__all_sync(0xffffffffu, nv == 32 || ncols == 0)) lse_chunk<32, kPoly>(rr, sl2, m, ssum);
              else if (nv > 0) lse_chunk_masked<32>(rr, nv, sl2, m, ssum);
            }
          }
          if (ncols > 0) leaf_row[(long long)leaf * G] = (m + lg2_approx(ssum)) * kLn2;
        }
      } else {
        const int4 st = s_up[i - n_leaf];
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
          uint32_t rr[32];
          tmem_ld_32x32(base + (uint32_t)(q * 32), rr);
          tmem_ld_wait();
          if (q == 3) handed_back();
          float* dst = up_row + st.z;
          const int node0 = st.y + ((q * 32) >> lgg);
          if (lgg == 1) score_nodes_g<2>(rr, sl2, G, head, dst, node0, st.w, live);
          else score_nodes_g<4>(rr, sl2, G, head, dst, node0, st.w, live);
        }
      }
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.status, (int)PISA_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, TM_COLS);
}

template <int D, int C, int NT>
int launch_dcn(const Geometry& g, const qm::Args& a, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
               const CUtensorMap& tm_p, int n_items, cudaStream_t s) {
  const size_t smem = (size_t)(D / 64) * 128 * 128 * (NT + score_stages(D, NT)) + 1024;
  return launch_dependent<qm_score_kernel<D, C, NT>>("qm_score", dim3((unsigned)n_items), 128 + 256 * NT, smem, s, g, a, tm_q, tm_k, tm_p);
}
template <int D, int C>
int launch_dc(const Geometry& g, const qm::Args& a, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
              const CUtensorMap& tm_p, cudaStream_t s) {
  if (a.tiles == 2) return launch_dcn<D, C, 2>(g, a, tm_q, tm_k, tm_p, a.n_items, s);
  return launch_dcn<D, C, 1>(g, a, tm_q, tm_k, tm_p, a.n_items, s);
}

}  // namespace

int launch_qm_score(const Geometry& g, const qm::Args& a, const void* q, const void* k, long long tokens, const void* pyramid,
                    long long pyr_rows, cudaStream_t s) {
  CUtensorMap tm_q, tm_k, tm_p;
  bool ok = qm_map_rows(&tm_q, q, g.d, g.Hq, tokens, g.B, g.qs, g.G, 128 / g.G);
  if (a.want_leaf) ok = ok && qm_map_rows(&tm_k, k, g.d, g.Hkv, tokens, g.B, g.ks, 1, 128);
  else tm_k = tm_q;                                         // never loaded from
  if (!ok) {
    record_cuda_error("qm_score tensor maps", cudaErrorInvalidValue);
    return PISA_ERR_CUDA;
  }
  {
    const uint64_t dims[3] = {(uint64_t)g.d, (uint64_t)pyr_rows, 1};
    const uint64_t str[3] = {2, (uint64_t)g.d * 2, (uint64_t)g.d * 2};
    const uint32_t box[3] = {64u, 128u, 1u};
    if (!tma::make_map(&tm_p, 2, 3, pyramid, dims, str, box, true)) {
      record_cuda_error("qm_score pyramid map", cudaErrorInvalidValue);
      return PISA_ERR_CUDA;
    }
  }
  if (g.d == 128) return g.C == 128 ? launch_dc<128, 128>(g, a, tm_q, tm_k, tm_p, s) : launch_dc<128, 64>(g, a, tm_q, tm_k, tm_p, s);
  return g.C == 128 ? launch_dc<64, 128>(g, a, tm_q, tm_k, tm_p, s) : launch_dc<64, 64>(g, a, tm_q, tm_k, tm_p, s);
}

// 4-D map of a [B, tokens, H, d] tensor (element strides b, n, h), one box = 64 columns of `heads` heads of `rows` tokens
bool qm_map_rows(void* map, const void* base, int d, int H, long long tokens, int B, const long long* st, int heads, int rows) {
  const uint64_t dims[4] = {(uint64_t)d, (uint64_t)H, (uint64_t)tokens, (uint64_t)B};
  const uint64_t str[4] = {2, (uint64_t)st[2] * 2, (uint64_t)st[1] * 2, (uint64_t)st[0] * 2};
  const uint32_t box[4] = {64u, (uint32_t)heads, (uint32_t)rows, 1u};
  return tma::make_map((CUtensorMap*)map, 2, 4, base, dims, str, box, true);
}

}  // namespace pisa
