// Leaf scoring of the level-2 nodes that a tile's rows share, query-major (shared.cuh).
//
// One item per tile of 128 / G tokens, drawn from a global counter: its queries stay in shared memory and the nodes of its list
// come by TMA tile loads, 256 keys a step (one node of 256 or two of 128 keys).  S = Q K^T as one chain of N = 256 UMMAs into
// one of two TMEM accumulators; two groups of eight epilogue warps take alternate steps, a warp 32 rows x 128 columns: the
// log-sum-exp of its leaf (C = 128) or two leaves (C = 64), written to the place the node has in the token's row.
// What bounds it: the exponentials, 128 x 256 a step = 2048 cycles of the special-function units, 85 % busy (a quarter of them on
// the FMA pipe: 4.96 ms instead of 4.80 at 65536 tokens, C = 128, 32 heads, half of a tile's tokens making a node shared); the
// tensor pipe's 1024 come second.  N = 256 because a chain of N = 128 instructions reads as many
// bytes of shared memory per clock as there are (operand A again for every instruction): 710 cycles instead of 512 a chain
// measured beside the loads.  The issuer looks at the next step's barriers before the last instructions of this one: it stands
// still while the pipe works, and the pipe while it does anything else.
// Rows that did not select a node take part in its products and are not stored; what is not finite in a key or query reaches
// only its own leaf's and row's score.  Every wait is bounded.
#include "lse_chunk.cuh"
#include "pisa_tensor.cuh"
#include "shared.cuh"
#include "tc_utils.cuh"
#include "tma_map.cuh"

namespace pisa {

using namespace tc;

namespace {

constexpr int kThreads = 640;
constexpr int kRing = 4;                       // items listed ahead
constexpr int kKeys = 256;                     // keys of a step

// How many of a tile's tokens make a node shared.  A step takes about 2450 cycles here (256 keys, 128 rows) at an SM clock of
// 1.7 GHz, in the lists a tile of gathered rows 3700 at 1.9 with nodes of 256 keys and 2840 with nodes of 128 (two of which are a
// step here).  Plan, inversion and both kernels in ms, lists alone and with 4 / 5 / 6 / 7 eighths of the tokens:
// 65536 tokens, C = 128, 32 heads: 6.78, 6.28 / 6.17 / 6.11 / 6.22; 32700, C = 64, fan-in 4, 32 heads: 1.72, 1.71 / 1.65 / 1.64 /
// 1.71; 40000, C = 64, fan-in 2, 16 heads: 0.99, 0.77 / 0.75 / 0.77 / 0.78; 65536, d = 64, 16 heads per group: 1.35, 1.19 / 1.19 /
// 1.19 / 1.19.
int share_threshold(const Geometry& g) { return (128 / g.G * (g.g * g.C == kKeys ? 6 : 5) + 7) / 8; }

struct ScoreArgs {
  SharedPlan plan;
  float* blk_lse;            // [BH, N, K * g, G]
  int32_t* ctr;
  int32_t* status;
  int n_items, fan;
};

// (max, sum of 2^(x - max)) over 64 columns in registers, x = raw * sl2
__device__ __forceinline__ void lse_64(const uint32_t (&a)[32], const uint32_t (&b)[32], float sl2, float& m, float& ssum) {
  float c[4];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    c[i] = __uint_as_float(a[i]);
    c[2 + i] = __uint_as_float(b[i]);
  }
#pragma unroll
  for (int j = 2; j < 30; j += 4) {
    c[0] = max3(c[0], __uint_as_float(a[j]), __uint_as_float(a[j + 1]));
    c[1] = max3(c[1], __uint_as_float(a[j + 2]), __uint_as_float(a[j + 3]));
    c[2] = max3(c[2], __uint_as_float(b[j]), __uint_as_float(b[j + 1]));
    c[3] = max3(c[3], __uint_as_float(b[j + 2]), __uint_as_float(b[j + 3]));
  }
  c[0] = max3(c[0], __uint_as_float(a[30]), __uint_as_float(a[31]));
  c[2] = max3(c[2], __uint_as_float(b[30]), __uint_as_float(b[31]));
  m = fmaxf(max3(c[0], c[1], c[2]), c[3]) * sl2;
  const uint64_t neg = pack2(-m, -m), sc = pack2(sl2, sl2);
  uint64_t s0 = pack2(0.f, 0.f), s1 = s0;
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    float x0, x1, y0, y1;
    unpack2(fma2(pack2(__uint_as_float(a[j]), __uint_as_float(a[j + 1])), sc, neg), x0, x1);
    unpack2(fma2(pack2(__uint_as_float(b[j]), __uint_as_float(b[j + 1])), sc, neg), y0, y1);
    s0 = add2(s0, pack2(ex2_approx(x0), ex2_approx(x1)));
    s1 = add2(s1, pack2(ex2_approx(y0), ex2_approx(y1)));
  }
  float p0, p1;
  unpack2(add2(s0, s1), p0, p1);
  ssum = p0 + p1;
}
// the same over the first nv (>= 1) of them
__device__ __forceinline__ void lse_64_masked(const uint32_t (&a)[32], const uint32_t (&b)[32], int nv, float sl2, float& m, float& ssum) {
  m = -CUDART_INF_F;
  ssum = 0.f;
  lse_chunk_masked<32>(a, min(nv, 32), sl2, m, ssum);
  if (nv > 32) lse_chunk_masked<32>(b, nv - 32, sl2, m, ssum);
}

__host__ __device__ constexpr int k_stages(int D) { return D == 128 ? 2 : 4; }

// NPS: nodes per step
template <int D, int C, int NPS>
__global__ void __launch_bounds__(kThreads, 1)
shared_score_kernel(Geometry geo, ScoreArgs a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = D / 64, A_SLAB = 128 * 128, B_SLAB = kKeys * 128, Q_TILE = KS * A_SLAB, K_TILE = KS * B_SLAB, NK = k_stages(D);
  constexpr int NODE = kKeys / NPS;            // keys of a node
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;                          // [2]
  uint8_t* sK = sQ + 2 * Q_TILE;               // [NK]
  __shared__ uint64_t q_full[2], q_empty[2], k_full[NK], k_empty[NK], t_full[2], t_empty[2], l_full[kRing], l_empty[kRing];
  __shared__ uint16_t s_node[kRing][kSharedMax];
  __shared__ int2 s_item[kRing];               // (work item or -1, its nodes)
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1);
      mbar_init(&t_full[i], 1); mbar_init(&t_empty[i], 8);
    }
    for (int i = 0; i < kRing; ++i) { mbar_init(&l_full[i], 1); mbar_init(&l_empty[i], 18); }
    for (int i = 0; i < NK; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1); }
    s_fail = 0;
    mbar_fence_init();
  }
  if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem = tmem_slot;             // accumulators at columns 0 and 256
  const int G = geo.G, lgG = 31 - __clz(G), tpt = 128 >> lgG, tiles = a.plan.tiles;

  auto next_item = [&](int it, int2& e) -> bool {
    const int r = it % kRing;
    if (!mbar_wait_bounded(&l_full[r], (uint32_t)((it / kRing) & 1))) { s_fail = 1; return false; }
    e = s_item[r];
    return e.x >= 0 && !s_fail;
  };
  auto done_item = [&](int it) {
    __syncwarp();
    if (lane == 0) mbar_arrive(&l_empty[it % kRing]);
  };

  if (warp == 3) {
    // ------------------------------------------------ scheduler
    for (int it = 0;; ++it) {
      const int r = it % kRing;
      bool ok = it < kRing || mbar_wait_bounded(&l_empty[r], (uint32_t)((it / kRing - 1) & 1));
      ok = __all_sync(0xffffffffu, ok && !s_fail);
      if (!ok) s_fail = 1;
      int item = a.n_items, n = 0;
      while (ok && n == 0) {                   // tiles that share nothing are left out
        if (lane == 0) item = atomicAdd(a.ctr, 1);
        item = __shfl_sync(0xffffffffu, item, 0);
        if (item >= a.n_items) break;
        n = min(a.plan.count[item], kSharedMax);
      }
      const bool more = ok && n > 0;
      if (more) {
        const uint16_t* src = a.plan.node + (long long)item * a.plan.max_nodes;
        for (int i = lane; i < n; i += 32) s_node[r][i] = src[i];
      }
      if (lane == 0) s_item[r] = make_int2(more ? item : -1, n);
      __syncwarp();
      if (lane == 0) mbar_arrive(&l_full[r]);
      if (!more) break;
    }
  } else if (warp == 0) {
    // ------------------------------------------------ TMA producer
    int ld = 0;
    int2 e;
    for (int it = 0; next_item(it, e); ++it) {
      const int bh = e.x / tiles, tile = e.x - bh * tiles, b = bh / geo.Hkv, h = bh % geo.Hkv;
      const int steps = (e.y + NPS - 1) / NPS;
      if (lane == 0) {
        const int qb = it & 1;
        bool ok = it < 2 || mbar_wait_bounded(&q_empty[qb], (uint32_t)(((it >> 1) - 1) & 1));
        if (ok) {
          mbar_arrive_expect_tx(&q_full[qb], (uint32_t)Q_TILE);
          for (int ks = 0; ks < KS; ++ks)
            tma_load_4d(smem_u32(sQ + qb * Q_TILE + ks * A_SLAB), &tm_q, &q_full[qb], ks * 64, h * G, tile * tpt, b);
        }
        for (int j = 0; j < steps && ok; ++j) {
          const int n = ld + j, st = n % NK;
          ok = n < NK || mbar_wait_bounded(&k_empty[st], (uint32_t)((n / NK - 1) & 1));
          if (!ok) break;
          mbar_arrive_expect_tx(&k_full[st], (uint32_t)K_TILE);
#pragma unroll
          for (int x = 0; x < NPS; ++x) {                          // (an odd list's last node twice)
            const int key = (int)s_node[it % kRing][min(j * NPS + x, e.y - 1)] * NODE;
            for (int ks = 0; ks < KS; ++ks)
              tma_load_4d(smem_u32(sK + st * K_TILE + ks * B_SLAB + x * (NODE * 128)), &tm_k, &k_full[st], ks * 64, h, key, b);
          }
        }
        if (!ok) s_fail = 1;
      }
      ld += steps;
      done_item(it);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ UMMA issuer (after a wait that gave up it runs through without waiting)
    const uint32_t idesc = make_idesc_bf16(128, kKeys, 0, 0);
    const uint32_t q_base = desc_lo(smem_u32(sQ), 0), k_base = desc_lo(smem_u32(sK), 0);
    bool dead = false;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (!dead && !mbar_try_wait(bar, parity) && !mbar_wait_bounded(bar, parity)) { dead = true; s_fail = 1; }
    };
    uint32_t k_st = 0u, k_ph = 0u, n = 0u;     // next stage and its phase; steps so far
    bool ready = false;
    int2 e;
    for (int it = 0; next_item(it, e); ++it) {
      const int ny = __shfl_sync(0xffffffffu, (e.y + NPS - 1) / NPS, 0);
      wait(&q_full[it & 1], (uint32_t)((it >> 1) & 1));
      const uint32_t q0 = q_base + (uint32_t)((it & 1) * (Q_TILE >> 4));
      for (int j = 0; j < ny; ++j, ++n) {
        const uint32_t buf = n & 1u;
        if (!ready) {
          wait(&k_full[k_st], k_ph);
          if (n >= 2u) wait(&t_empty[buf], ((n >> 1) - 1u) & 1u);
        }
        tcgen05_fence_after_sync();
        const uint32_t d0 = tmem + buf * (uint32_t)kKeys, k0 = k_base + k_st * (uint32_t)(K_TILE >> 4);
        auto mma = [&](int kk) {
          umma_bf16(d0, desc64(q0 + ((uint32_t)((kk >> 2) * A_SLAB + (kk & 3) * 32) >> 4)),
                    desc64(k0 + ((uint32_t)((kk >> 2) * B_SLAB + (kk & 3) * 32) >> 4)), idesc, kk > 0);
        };
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16 - 1; ++kk) mma(kk);
        }
        __syncwarp();
        const uint32_t k_nx = (k_st + 1 == (uint32_t)NK) ? 0u : k_st + 1, k_nph = k_ph ^ (k_nx == 0u ? 1u : 0u);
        ready = mbar_test(&k_full[k_nx], k_nph) & (n == 0u || mbar_test(&t_empty[buf ^ 1u], (((n + 1u) >> 1) - 1u) & 1u));
        if (elect_one()) {
          mma(D / 16 - 1);
          umma_commit(&t_full[buf]);
          umma_commit(&k_empty[k_st]);
        }
        __syncwarp();
        k_st = k_nx;
        k_ph = k_nph;
      }
      if (elect_one()) umma_commit(&q_empty[it & 1]);
      done_item(it);
    }
  } else if (warp >= 4) {
    // ------------------------------------------------ epilogue
    const int grp = (warp - 4) >> 3, cg = ((warp - 4) >> 2) & 1, quarter = warp & 3;
    const int row = quarter * 32 + lane, head = row & (G - 1), tl = row >> lgG;
    const uint32_t base = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(grp * kKeys + cg * 128);
    const float sl2 = geo.scale * kLog2e;
    const int fan = a.fan, x0 = (NPS == 2) ? cg : 0;                 // this warp's node of a step
    int kv = 0, cnt = 0;                                             // steps of the items before; steps of this group
    int2 e;
    for (int it = 0; next_item(it, e); ++it) {
      const int bh = e.x / tiles, tile = e.x - bh * tiles;
      const int t = tile * tpt + tl, ny = (e.y + NPS - 1) / NPS, c_t = t / C;
      const uint16_t* list = s_node[it % kRing];
      const uint8_t* slots = a.plan.slot + (long long)e.x * a.plan.max_nodes * tpt + tl;
      float* dst = a.blk_lse + ((long long)bh * geo.N + t) * (geo.K * fan) * G + head;
      auto slot_of = [&](int j) -> int { return (j < ny && j * NPS + x0 < e.y) ? (int)slots[(j * NPS + x0) * tpt] : 255; };
      bool ok = true;
      int j = (kv ^ grp) & 1;
      int slot_next = slot_of(j);
      for (; j < ny && ok; j += 2, ++cnt) {
        const int slot = slot_next, node = (int)list[min(j * NPS + x0, e.y - 1)];
        slot_next = slot_of(j + 2);                                  // in flight during this step
        const bool sel = slot != 255;
        ok = mbar_wait_bounded(&t_full[grp], (uint32_t)(cnt & 1));
        if (!ok) break;
        tcgen05_fence_after_sync();
        const bool any = __any_sync(0xffffffffu, sel);
        float m[2], ssum[2];                                         // of the two 64-column halves
        // leaf of a half: C = 128: the warp's one; C = 64: one each (a node of 128 keys is this warp's alone)
        const int leaf0 = node * fan + (C == 128 ? cg : NPS == 2 ? 0 : cg * 2);
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          uint32_t ra[32], rb[32];
          if (any) {
            tmem_ld_32x32(base + (uint32_t)(hh * 64), ra);
            tmem_ld_32x32(base + (uint32_t)(hh * 64 + 32), rb);
            tmem_ld_wait();
          }
          if (hh == 1) {                                             // the accumulator is in registers
            tcgen05_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(&t_empty[grp]);
          }
          if (any) {
            const int leaf = leaf0 + (C == 64 ? hh : 0);
            int ncols = 0;                                           // causally visible columns of the leaf for this row
            if (sel && leaf <= c_t && leaf < geo.M[1]) ncols = (leaf == c_t) ? t - leaf * C + 1 : min(C, geo.N - leaf * C);
            const int nv = max(0, min(64, ncols - (C == 128 ? hh * 64 : 0)));
            m[hh] = -CUDART_INF_F;
            ssum[hh] = 0.f;
            if (__all_sync(0xffffffffu, nv == 64 || nv == 0)) {
              if (__any_sync(0xffffffffu, nv > 0)) {
                float mm, ss;
                lse_64(ra, rb, sl2, mm, ss);
                if (nv > 0) { m[hh] = mm; ssum[hh] = ss; }
              }
            } else if (nv > 0) {
              lse_64_masked(ra, rb, nv, sl2, m[hh], ssum[hh]);
            }
            if (C == 64 && sel) dst[(slot * fan + (leaf - node * fan)) * G] = ncols > 0 ? (m[hh] + log2f(ssum[hh])) * kLn2 : -CUDART_INF_F;
          }
        }
        if (C == 128 && any && sel) {
          float mm = m[0], ss = ssum[0];
          if (ssum[1] != 0.f) {                                      // (0: no visible column; NaN takes part)
            mm = fmaxf(m[0], m[1]);
            ss = (m[0] == mm ? ssum[0] : ssum[0] * ex2_approx(m[0] - mm)) + (m[1] == mm ? ssum[1] : ssum[1] * ex2_approx(m[1] - mm));
          }
          dst[(slot * fan + cg) * G] = ss != 0.f ? (mm + log2f(ss)) * kLn2 : -CUDART_INF_F;
        }
      }
      kv += ny;
      if (!ok) s_fail = 1;
      done_item(it);
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.status, (int)PISA_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, 512);
}

template <int D, int C, int NPS>
int launch_dcn(const Geometry& g, const ScoreArgs& a, const CUtensorMap& tm_q, const CUtensorMap& tm_k, cudaStream_t s) {
  const size_t smem = (size_t)(D / 64) * (2 * 128 + k_stages(D) * kKeys) * 128 + 1024;
  const cudaError_t e = cudaFuncSetAttribute(shared_score_kernel<D, C, NPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) { record_cuda_error("shared_score attr", e); return PISA_ERR_CUDA; }
  const int grid = a.n_items < num_sms() ? a.n_items : num_sms();
  shared_score_kernel<D, C, NPS><<<grid, kThreads, smem, s>>>(g, a, tm_q, tm_k);
  return check_launch("shared_score");
}
template <int D>
int launch_d(const Geometry& g, const ScoreArgs& a, const CUtensorMap& tm_q, const CUtensorMap& tm_k, cudaStream_t s) {
  if (g.C == 128) return launch_dcn<D, 128, 1>(g, a, tm_q, tm_k, s);       // fan-in 2
  return g.g == 2 ? launch_dcn<D, 64, 2>(g, a, tm_q, tm_k, s) : launch_dcn<D, 64, 1>(g, a, tm_q, tm_k, s);
}

}  // namespace

size_t shared_score_layout(const Geometry& g, char* ws, SharedPlan* p) {
  const int tpt = 128 / g.G;
  const size_t bh = (size_t)g.B * g.Hkv;
  if (g.g * g.C != 256 && !(g.g == 2 && g.C == 64)) return SIZE_MAX;
  p->threshold = share_threshold(g);
  p->span = g.C * g.g;
  p->words = 0;
  p->tiles = (g.N + tpt - 1) / tpt;
  const int most = g.K * tpt / p->threshold;
  p->max_nodes = most < kSharedMax ? most : kSharedMax;
  const size_t tiles = bh * p->tiles;
  size_t o = 0;
  auto take = [&](size_t bytes) { char* r = ws + o; o += align_up(bytes, 4); return r; };
  p->taken = (uint32_t*)take(bh * g.N * 4);
  p->count = (int32_t*)take(tiles * 4);
  p->node = (uint16_t*)take(tiles * p->max_nodes * 2);
  p->slot = (uint8_t*)take(tiles * p->max_nodes * tpt);
  p->mask = nullptr;
  p->chain = nullptr;
  return o;
}

int launch_shared_score(const Geometry& g, const void* q, const void* k, float* blk_lse, const SharedPlan& plan, int32_t* ctr,
                        int32_t* status, cudaStream_t s) {
  CUtensorMap tm_q, tm_k;
  if (!qm_map_rows(&tm_q, q, g.d, g.Hq, g.N, g.B, g.qs, g.G, 128 / g.G) || !qm_map_rows(&tm_k, k, g.d, g.Hkv, g.N, g.B, g.ks, 1, g.g * g.C)) {
    record_cuda_error("shared_score tensor maps", cudaErrorInvalidValue);
    return PISA_ERR_CUDA;
  }
  ScoreArgs a;
  a.plan = plan;
  a.blk_lse = blk_lse; a.ctr = ctr; a.status = status;
  a.n_items = g.B * g.Hkv * plan.tiles;
  a.fan = g.g;
  return g.d == 128 ? launch_d<128>(g, a, tm_q, tm_k, s) : launch_d<64>(g, a, tm_q, tm_k, s);
}

}  // namespace pisa
