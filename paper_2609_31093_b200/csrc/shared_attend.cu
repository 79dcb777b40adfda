// Attention over the leaves that a tile's rows share, query-major (shared.cuh).
//
// The lists cost about 5000 SM cycles per 128-row tile of gathered (token, leaf) pairs (C = 128; 4300 with C = 64), most of it
// for the fp32 rows added into memory; a dense step here costs a third of that and adds nothing into memory.  One item per
// tile, drawn from a global counter: its queries stay in shared memory, the leaves of its list come by TMA tile loads, 128 keys
// a step (one leaf of 128 or two of 64 keys, wherever they lie); S = Q K^T -> P = exp(S - lse) in bf16 where selected and
// visible, zero elsewhere (the row's denominator is known from the routing, so P is final), over S in TMEM -> O += P V.  The
// accumulator rows are STORED: nothing clears them first, the list-driven kernel then adds to them.
// Roles: warp 0 loads queries and keys, warp 2 values, warp 1 issues the products, warp 3 draws the items, warps 4-11 and
// 12-19 are two softmax / read-out groups on alternate steps; inside a group two warps share a TMEM lane quarter, half of the
// columns each.  Three S / P buffers, so that a step's softmax has the products of two others to run under.
// Measured: 131072 tokens, 32 heads, C = 128: 6.6 ms for 77 % of the routed pairs and the forced leaves, 1660 cycles a step,
// 1230 TFLOP/s executed (three quarters of the measured bf16 peak; the SM clock falls to 1.65 GHz); the lists take 16.8 ms for all
// of the routed pairs.
// Every wait is bounded.  What is not finite reaches only the rows that selected it: rows that came out not finite are
// computed again from their own leaves (attend_shared_row).
#include "shared.cuh"

#include "lse_chunk.cuh"
#include "pisa_tensor.cuh"
#include "tc_utils.cuh"
#include "tma_map.cuh"

namespace pisa {

using namespace tc;

namespace {

constexpr int kThreads = 640;
constexpr int kRing = 4;                       // items listed ahead: reading an item out waits for products that go out two items later
constexpr int kBufs = 3;                       // S / P buffers
// How many of a tile's tokens make a leaf shared.  A dense step takes about 1660 cycles of an SM (128 keys; 128 rows, d = 128)
// whoever selected its leaves, 32 tokens' pairs with a leaf (G = 4) 5000 in the lists with C = 128 and 4300 with C = 64, and
// without groups the lists' reductions are scalar.  Plan, shared and list attention in ms, by sixteenths: 131072 tokens,
// C = 128: 4: 11.42, 6: 11.39, 8: 11.35; 2 x 32700, C = 64, G = 4: 4: 2.08, 6: 2.18, 8: 2.30; 40000, C = 64, G = 1: 4: 1.70,
// 6: 1.88, 8: 2.08.
int share_threshold(const Geometry& g) {
  const int tpt = 128 / g.G, num = g.C == 128 ? 6 : (g.G == 1 ? 3 : 4);
  return (tpt * num + 15) / 16;
}

template <bool V> struct Bool { static constexpr bool value = V; };

// ------------------------------------------------------------------ attention

struct AttArgs {
  SharedPlan plan;
  const float* row_lse;      // [B, Hq, N] natural log
  const __nv_bfloat16 *q, *k, *v;   // for attend_shared_row()
  float* o_acc;              // fp32: [B, Hkv, N, 128, G] for d = 128, [B, N, Hq, 64] for d = 64 (the layouts of pv_ws)
  int32_t* ctr;
  int32_t* status;
  int n_items;
};

// One row over its own shared leaves only, by one warp (`sel`: does the row's token have the leaf at this place of the list).
template <int D, typename SEL>
__device__ __forceinline__ void attend_shared_row(const __nv_bfloat16* q, const __nv_bfloat16* k, long long ks, const __nv_bfloat16* v,
                                                  long long vs, const uint16_t* leaves, int n, SEL sel, int t, int C, float sl2,
                                                  float neg_lse2, float* out, int out_stride) {
  const int lane = threadIdx.x & 31;
  float acc[D / 32];
#pragma unroll
  for (int y = 0; y < D / 32; ++y) acc[y] = 0.f;
  for (int i = 0; i < n; ++i) {
    if (!sel(i)) continue;
    const int leaf = leaves[i], end = min((leaf + 1) * C, t + 1);
    for (int j0 = leaf * C; j0 < end; j0 += 32) {
      const int j = j0 + lane;
      float p = 0.f;
      if (j < end) {
        float s = 0.f;
#pragma unroll 4
        for (int c = 0; c < D; c += 8) {
          float x[8], y[8];
          Elem<__nv_bfloat16>::load_chunk(q + c, x);
          Elem<__nv_bfloat16>::load_chunk(k + j * ks + c, y);
#pragma unroll
          for (int e = 0; e < 8; ++e) s = fmaf(x[e], y[e], s);
        }
        p = __bfloat162float(__float2bfloat16_rn(ex2_approx(fmaf(s, sl2, neg_lse2))));
      }
      for (int x = 0; x < min(32, end - j0); ++x) {
        const float px = __shfl_sync(0xffffffffu, p, x);
#pragma unroll
        for (int y = 0; y < D / 32; ++y) acc[y] = fmaf(px, __bfloat162float(v[(long long)(j0 + x) * vs + lane + 32 * y]), acc[y]);
      }
    }
  }
#pragma unroll
  for (int y = 0; y < D / 32; ++y) out[(long long)(lane + 32 * y) * out_stride] = acc[y];
}

// Tiles of 128 keys / values in flight: what two query tiles leave of 227 KB.  A step's keys are needed three steps before its
// values, so the two have rings (and loading warps) of their own.
__host__ __device__ constexpr int k_stages(int D) { return D == 128 ? 2 : 4; }
__host__ __device__ constexpr int v_stages(int D) { return D == 128 ? 3 : 6; }

template <int D, int C>
__global__ void __launch_bounds__(kThreads, 1)
shared_attend_kernel(Geometry geo, AttArgs a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                     const __grid_constant__ CUtensorMap tm_v) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = D / 64, SLAB = 128 * 128, TILE = KS * SLAB, NK = k_stages(D), NV = v_stages(D);
  constexpr int LPS = 128 / C;               // leaves per step
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;                        // [2] query tiles of this item and the next
  uint8_t* sK = sQ + 2 * TILE;               // [NK]
  uint8_t* sV = sK + NK * TILE;              // [NV]
  __shared__ uint64_t q_full[2], q_empty[2], k_full[NK], k_empty[NK], v_full[NV], v_empty[NV], s_full[kBufs], p_full[kBufs],
      o_full, o_empty, l_full[kRing], l_empty[kRing];
  __shared__ uint16_t s_leaf[kRing][kSharedMax];
  __shared__ int2 s_item[kRing];             // (work item or -1, its leaves)
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  __shared__ volatile int s_again;           // some row came out not finite
  __shared__ volatile int s_items;           // this CTA's items: the last one + 1 (the others: plan.chain)

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1); }
    for (int i = 0; i < kRing; ++i) { mbar_init(&l_full[i], 1); mbar_init(&l_empty[i], 19); }
    for (int i = 0; i < kBufs; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 8); }
    mbar_init(&o_full, 1); mbar_init(&o_empty, 16);
    for (int i = 0; i < NK; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1); }
    for (int i = 0; i < NV; ++i) { mbar_init(&v_full[i], 1); mbar_init(&v_empty[i], 1); }
    s_fail = 0;
    s_again = 0;
    s_items = 0;
    mbar_fence_init();
  }
  if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem = tmem_slot;           // S / P buffers at columns 0, 128, 256, O at 384
  const int G = geo.G, lgG = 31 - __clz(G), tpt = 128 >> lgG, tiles = a.plan.tiles;

  // the next ring entry: false when there is no more work (or something failed)
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
      int item = 0;
      if (lane == 0) item = ok ? atomicAdd(a.ctr, 1) : a.n_items;
      item = __shfl_sync(0xffffffffu, item, 0);
      const bool more = ok && item < a.n_items;
      int n = 0;
      if (more) {
        n = min(a.plan.count[item], kSharedMax);
        const uint16_t* src = a.plan.node + (long long)item * a.plan.max_nodes;
        for (int i = lane; i < n; i += 32) s_leaf[r][i] = src[i];
      }
      if (lane == 0) {
        s_item[r] = make_int2(more ? item : -1, n);
        if (more) {
          a.plan.chain[item] = s_items;
          s_items = item + 1;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&l_full[r]);
      if (!more) break;
    }
  } else if (warp == 0 || warp == 2) {
    // ------------------------------------------------ TMA producers: queries and keys; values
    // (a warp each: the values' stages come free one product later than the keys', and the next keys would wait behind that)
    int ld = 0;                                                    // steps loaded so far
    int2 e;
    for (int it = 0; next_item(it, e); ++it) {
      const int bh = e.x / tiles, tile = e.x - bh * tiles, b = bh / geo.Hkv, h = bh % geo.Hkv;
      const int steps = (e.y + LPS - 1) / LPS;
      if (lane == 0) {
        bool ok = true;
        if (warp == 0) {
          const int qb = it & 1;
          ok = it < 2 || mbar_wait_bounded(&q_empty[qb], (uint32_t)(((it >> 1) - 1) & 1));
          if (ok) {
            mbar_arrive_expect_tx(&q_full[qb], (uint32_t)TILE);
            for (int ks = 0; ks < KS; ++ks)
              tma_load_4d(smem_u32(sQ + qb * TILE + ks * SLAB), &tm_q, &q_full[qb], ks * 64, h * G, tile * tpt, b);
          }
        }
        uint64_t* full = (warp == 0) ? k_full : v_full;
        uint64_t* empty = (warp == 0) ? k_empty : v_empty;
        uint8_t* dst = (warp == 0) ? sK : sV;
        const void* map = (warp == 0) ? (const void*)&tm_k : (const void*)&tm_v;
        const int ns = (warp == 0) ? NK : NV;
        for (int j = 0; j < steps && ok; ++j) {
          const int n = ld + j, st = n % ns;
          ok = n < ns || mbar_wait_bounded(&empty[st], (uint32_t)((n / ns - 1) & 1));
          if (!ok) break;
          mbar_arrive_expect_tx(&full[st], (uint32_t)TILE);
#pragma unroll
          for (int x = 0; x < LPS; ++x) {                          // (an odd list's last leaf twice: nobody selected the second one)
            const int key = (int)s_leaf[it % kRing][min(j * LPS + x, e.y - 1)] * C;
            for (int ks = 0; ks < KS; ++ks)
              tma_load_4d(smem_u32(dst + st * TILE + ks * SLAB + x * (C * 128)), map, &full[st], ks * 64, h, key, b);
          }
        }
        if (!ok) s_fail = 1;
      }
      ld += steps;
      done_item(it);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ UMMA issuer
    // An instruction is taken when the tensor pipe has room for it: this warp stands still while the pipe works, and the pipe
    // while the warp does anything else.  So a step's two chains go out as one run, and the barriers of the next step are
    // looked at before its last instructions (a wait before each chain: 2160 cycles a step, of them 1090 in the chains,
    // whether the softmax ran or not).  After a wait that gave up the loop runs through without waiting (its operands stay
    // inside this CTA's memory) and the status word tells.
    const uint32_t idesc_s = make_idesc_bf16(128, 128, 0, 0);
    const uint32_t idesc_o = make_idesc_bf16(128, D, 0, 1);
    const uint32_t q_base = desc_lo(smem_u32(sQ), 0), k_base = desc_lo(smem_u32(sK), 0), v_base = desc_lo(smem_u32(sV), SLAB);
    bool dead = false;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (!dead && !mbar_try_wait(bar, parity) && !mbar_wait_bounded(bar, parity)) { dead = true; s_fail = 1; }
    };
    // steps whose S is out and whose product of P with the values is owed: 0 = none, else bit 0 and bit 1 = first / last of its item
    uint32_t owed[kBufs];
#pragma unroll
    for (int i = 0; i < kBufs; ++i) owed[i] = 0u;
    uint32_t pv_buf = 0u, pv_ph = 0u, v_st = 0u, v_ph = 0u, n_out = 0u;   // of the next product: buffer, stage, their phases; outputs begun
    uint32_t k_st = 0u, k_ph = 0u, sb = 0u;                         // next stage of keys, its phase; next S buffer
    auto wait_product = [&](uint32_t w, bool ready) {
      if (!ready) {
        wait(&p_full[pv_buf], pv_ph);
        wait(&v_full[v_st], v_ph);
      }
      if ((w & 1u) && n_out++ > 0u) wait(&o_empty, n_out & 1u);
    };
    auto issue_product = [&](uint32_t w) {                          // (by the elected lane)
      const uint32_t p0 = tmem + pv_buf * 128u, d0 = tmem + kBufs * 128u, v0 = v_base + v_st * (uint32_t)(TILE >> 4);
      const uint32_t acc = (w & 1u) ? 0u : 1u;
#pragma unroll
      for (int kk = 0; kk < 8; ++kk)                                // sixteen keys: eight columns of P, its halves 64 apart
        umma_bf16_ts(d0, p0 + (uint32_t)((kk >> 2) * 64 + (kk & 3) * 8), desc64(v0 + kk * (2048 >> 4)), idesc_o, kk > 0 ? 1u : acc);
      umma_commit(&v_empty[v_st]);
      if (w & 2u) umma_commit(&o_full);
    };
    auto next_product = [&]() {
      if (++pv_buf == (uint32_t)kBufs) { pv_buf = 0u; pv_ph ^= 1u; }
      if (++v_st == (uint32_t)NV) { v_st = 0u; v_ph ^= 1u; }
    };
    auto issue_scores = [&](uint32_t q0, int kk) {
      const uint32_t o = (uint32_t)((kk >> 2) * SLAB + (kk & 3) * 32) >> 4;
      umma_bf16(tmem + sb * 128u, desc64(q0 + o), desc64(k_base + k_st * (uint32_t)(TILE >> 4) + o), idesc_s, kk > 0);
    };
    constexpr int HOLD = (D == 128) ? 3 : 1;                        // instructions still to go out when the next step is looked at
    bool p_ready = false, k_ready = false;
    int2 e;
    for (int it = 0; next_item(it, e); ++it) {
      const int ny = __shfl_sync(0xffffffffu, (e.y + LPS - 1) / LPS, 0);
      wait(&q_full[it & 1], (uint32_t)((it >> 1) & 1));
      const uint32_t q0 = q_base + (uint32_t)((it & 1) * (TILE >> 4));
      for (int j = 0; j < ny; ++j) {
        const uint32_t w = owed[0];                                 // the one whose P stands in this step's buffer
        if (w != 0u) wait_product(w, p_ready);
        if (!k_ready) wait(&k_full[k_st], k_ph);
        tcgen05_fence_after_sync();
        if (elect_one()) {
          if (w != 0u) issue_product(w);
#pragma unroll
          for (int kk = 0; kk < D / 16 - HOLD; ++kk) issue_scores(q0, kk);
        }
        __syncwarp();
        if (w != 0u) next_product();
        const uint32_t k_nx = (k_st + 1 == (uint32_t)NK) ? 0u : k_st + 1, k_nph = k_ph ^ (k_nx == 0u ? 1u : 0u);
        k_ready = mbar_test(&k_full[k_nx], k_nph);
        p_ready = mbar_test(&p_full[pv_buf], pv_ph) & mbar_test(&v_full[v_st], v_ph);
        if (elect_one()) {
#pragma unroll
          for (int kk = D / 16 - HOLD; kk < D / 16; ++kk) issue_scores(q0, kk);
          umma_commit(&s_full[sb]);
          umma_commit(&k_empty[k_st]);
        }
        __syncwarp();
#pragma unroll
        for (int i = 0; i + 1 < kBufs; ++i) owed[i] = owed[i + 1];
        owed[kBufs - 1] = 4u | (j == 0 ? 1u : 0u) | (j == ny - 1 ? 2u : 0u);
        if (++sb == (uint32_t)kBufs) sb = 0u;
        k_st = k_nx;
        k_ph = k_nph;
      }
      if (elect_one()) umma_commit(&q_empty[it & 1]);
      done_item(it);
    }
#pragma unroll
    for (int u = 0; u < kBufs; ++u)                                 // what is still owed, older steps first
      if (owed[u] != 0u) {
        wait_product(owed[u], false);
        tcgen05_fence_after_sync();
        if (elect_one()) issue_product(owed[u]);
        __syncwarp();
        next_product();
      }
  } else if (warp >= 4) {
    // ------------------------------------------------ softmax and read-out
    const int grp = (warp - 4) >> 3, half = ((warp - 4) >> 2) & 1, quarter = warp & 3;
    const int row = quarter * 32 + lane, head = row & (G - 1), tl = row >> lgG;
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    const float sl2 = geo.scale * kLog2e;
    const int MW = a.plan.words;
    int kv = 0;                                  // steps of the items before this one
    constexpr int HC = D / 4;                    // output columns of one warp
    const int col0 = (grp * 2 + half) * HC;
    float* out_row = nullptr;                    // accumulator of the item that is still to be read out (null: no such row)
    int outs = 0;
    auto read_out = [&]() -> bool {
      if (!mbar_wait_bounded(&o_full, (uint32_t)(outs & 1))) { s_fail = 1; return false; }
      ++outs;
      tcgen05_fence_after_sync();
      const uint32_t o_base = tmem + lane_sel + (uint32_t)(kBufs * 128 + col0);
      uint32_t rr[HC];
      if constexpr (HC == 32) tmem_ld_32x32(o_base, rr);
      else tmem_ld_32x16(o_base, rr);
      tmem_ld_wait();
      tcgen05_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&o_empty);
      uint64_t finite[2] = {0ull, 0ull};                                     // NaN once a value is infinite or NaN
#pragma unroll
      for (int x = 0; x < HC / 2; ++x)
        finite[x & 1] = fma2(pack2(__uint_as_float(rr[2 * x]), __uint_as_float(rr[2 * x + 1])), 0ull, finite[x & 1]);
      float f0, f1;
      unpack2(add2(finite[0], finite[1]), f0, f1);
      if (out_row != nullptr && f0 + f1 != 0.f) s_again = 1;
      if (D == 64 || G == 1) {
        // the row's columns are adjacent
        if (out_row != nullptr)
#pragma unroll
          for (int i = 0; i < HC; i += 4)
            *reinterpret_cast<float4*>(out_row + col0 + i) = make_float4(__uint_as_float(rr[i]), __uint_as_float(rr[i + 1]),
                                                                        __uint_as_float(rr[i + 2]), __uint_as_float(rr[i + 3]));
      } else if (G == 2) {
        // [d][2]: two lanes (the heads of a token) exchange, each stores both heads of every other column
        const bool up = (lane & 1) != 0;
#pragma unroll
        for (int i = 0; i < HC; i += 2) {
          const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? rr[i] : rr[i + 1], 1);
          const uint32_t x = up ? got : rr[i], y = up ? rr[i + 1] : got;
          if (out_row != nullptr)
            *reinterpret_cast<float2*>(out_row - head + (col0 + i + (up ? 1 : 0)) * 2) = make_float2(__uint_as_float(x), __uint_as_float(y));
        }
      } else {
        // [d][G]: four lanes (four heads of a token) transpose 4 x 4, each stores the four heads of every fourth column
        const bool u1 = (lane & 1) != 0, u2 = (lane & 2) != 0;
#pragma unroll
        for (int i = 0; i < HC; i += 4) {
          const uint32_t g0 = __shfl_xor_sync(0xffffffffu, u1 ? rr[i] : rr[i + 1], 1), g1 = __shfl_xor_sync(0xffffffffu, u1 ? rr[i + 2] : rr[i + 3], 1);
          const uint32_t n0 = u1 ? g0 : rr[i], n1 = u1 ? rr[i + 1] : g0, n2 = u1 ? g1 : rr[i + 2], n3 = u1 ? rr[i + 3] : g1;
          const uint32_t h0 = __shfl_xor_sync(0xffffffffu, u2 ? n0 : n2, 2), h1 = __shfl_xor_sync(0xffffffffu, u2 ? n1 : n3, 2);
          if (out_row != nullptr)
            *reinterpret_cast<float4*>(out_row - (head & 3) + (long long)(col0 + i + (lane & 3)) * G) =
                make_float4(__uint_as_float(u2 ? h0 : n0), __uint_as_float(u2 ? h1 : n1), __uint_as_float(u2 ? n2 : h0),
                            __uint_as_float(u2 ? n3 : h1));
        }
      }
      return true;
    };
    int2 e;
    for (int it = 0; next_item(it, e); ++it) {
      const int bh = e.x / tiles, tile = e.x - bh * tiles, b = bh / geo.Hkv, h = bh % geo.Hkv;
      const int t = tile * tpt + tl, ny = (e.y + LPS - 1) / LPS;
      const bool live = t < geo.N;
      const uint16_t* list = s_leaf[it % kRing];
      const uint32_t* masks = a.plan.mask + (long long)e.x * a.plan.max_nodes * MW + (tl >> 5);
      float neg_lse2 = 0.f;
      if (live) neg_lse2 = -a.row_lse[((long long)b * geo.Hq + h * G + head) * geo.N + t] * kLog2e;
      bool ok = true, owes = it > 0;             // owes: the item before this one is still to be read out
      const int x0 = (C == 64) ? half : 0;       // this warp's leaf of a step
      auto mask_of = [&](int j) -> uint32_t { return (j < ny && j * LPS + x0 < e.y) ? masks[(j * LPS + x0) * MW] : 0u; };
      int j = (kv ^ grp) & 1;                    // this group's first step of the item
      uint32_t word = mask_of(j);
      for (; j < ny && ok; j += 2) {
        const bool sel = live && ((word >> (tl & 31)) & 1u);
        const int key0 = (int)list[min(j * LPS + x0, e.y - 1)] * C + (C == 64 ? 0 : half * 64);
        word = mask_of(j + 2);                   // in flight during this step
        const int n = kv + j, buf = n % kBufs;
        const uint32_t s_base = tmem + lane_sel + (uint32_t)(buf * 128 + half * 64);   // this warp's columns of S, then of P
        ok = mbar_wait_bounded(&s_full[buf], (uint32_t)((n / kBufs) & 1));
        if (!ok) break;
        tcgen05_fence_after_sync();
        const int nv = sel ? max(0, min(64, t - key0 + 1)) : 0;      // keys of these 64 the row selected and may see
        // (two bodies: a warp whose rows see all of their leaves -- nearly every one -- does without two instructions per key)
        auto probs = [&](int qq, auto masked) {
          const float bias = sel ? neg_lse2 : -CUDART_INF_F;                 // exp2(-inf) = 0: the row did not select the leaf
          const uint64_t sc2 = pack2(sl2, sl2), bias2 = pack2(bias, bias);
          uint32_t rr[32], pk[16];
          tmem_ld_32x32(s_base + (uint32_t)(qq * 32), rr);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 16; ++x) {
            float z0, z1;
            unpack2(fma2(pack2(__uint_as_float(rr[2 * x]), __uint_as_float(rr[2 * x + 1])), sc2, bias2), z0, z1);
            float p0 = ex2_approx(z0), p1 = ex2_approx(z1);
            if (masked.value) {
              if (qq * 32 + 2 * x >= nv) p0 = 0.f;
              if (qq * 32 + 2 * x + 1 >= nv) p1 = 0.f;
            }
            const __nv_bfloat162 pp = __floats2bfloat162_rn(p0, p1);
            pk[x] = *reinterpret_cast<const uint32_t*>(&pp);
          }
          tmem_st_32x16(s_base + (uint32_t)(qq * 16), pk);                   // over columns of S this warp has already read
        };
        if (__any_sync(0xffffffffu, nv > 0)) {
          if (__all_sync(0xffffffffu, nv == 64 || !sel)) {
            probs(0, Bool<false>());
            probs(1, Bool<false>());
          } else {
            probs(0, Bool<true>());
            probs(1, Bool<true>());
          }
        } else {
          uint32_t pk[16];
#pragma unroll
          for (int x = 0; x < 16; ++x) pk[x] = 0u;
          tmem_st_32x16(s_base, pk);
          tmem_st_32x16(s_base + 16u, pk);
        }
        tmem_st_wait();
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[buf]);
        if (owes) {                                 // (behind this item's first probabilities, so that the tensor pipe has work)
          ok = read_out();
          owes = false;
        }
      }
      if (ok && owes) ok = read_out();
      kv += ny;
      if (!ok) s_fail = 1;
      done_item(it);
      const long long unit_row = (long long)bh * geo.N + t;
      out_row = !live ? nullptr
                      : (D == 128) ? a.o_acc + unit_row * (D * G) + head : a.o_acc + (((long long)b * geo.N + t) * geo.Hq + h * G + head) * D;
    }
    if (kv > 0 && !s_fail) read_out();
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.status, (int)PISA_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, 512);
  if (!s_again || s_fail) return;
  for (int item = s_items - 1; item >= 0; item = a.plan.chain[item] - 1) {
    const int bh = item / tiles, tile = item - bh * tiles, h = bh % geo.Hkv;
    const long long b = bh / geo.Hkv;
    for (int row = warp; row < 128; row += kThreads / 32) {
      const int tl = row >> lgG, t = tile * tpt + tl, head = row & (G - 1), hq = h * G + head;
      if (t >= geo.N) break;
      const int stride = (D == 128) ? G : 1;
      float* out = (D == 128) ? a.o_acc + ((long long)bh * geo.N + t) * (D * G) + head : a.o_acc + ((b * geo.N + t) * geo.Hq + hq) * D;
      float finite = 0.f;
#pragma unroll
      for (int y = 0; y < D / 32; ++y) finite = fmaf(out[(long long)(lane + 32 * y) * stride], 0.f, finite);
      if (!__any_sync(0xffffffffu, finite != finite)) continue;
      const uint32_t* masks = a.plan.mask + (long long)item * a.plan.max_nodes * a.plan.words + (tl >> 5);
      attend_shared_row<D>(a.q + b * geo.qs[0] + t * geo.qs[1] + hq * geo.qs[2], a.k + b * geo.ks[0] + h * geo.ks[2], geo.ks[1],
                           a.v + b * geo.vs[0] + h * geo.vs[2], geo.vs[1], a.plan.node + (long long)item * a.plan.max_nodes,
                           a.plan.count[item], [&](int i) { return ((masks[i * a.plan.words] >> (tl & 31)) & 1u) != 0u; }, t, C,
                           geo.scale * kLog2e, -a.row_lse[(b * geo.Hq + hq) * geo.N + t] * kLog2e, out, stride);
    }
  }
}

template <int D, int C>
int launch_dc(const Geometry& g, const AttArgs& a, const CUtensorMap& tm_q, const CUtensorMap& tm_k, const CUtensorMap& tm_v,
              cudaStream_t s) {
  const size_t smem = (size_t)(D / 64) * (2 + k_stages(D) + v_stages(D)) * 128 * 128 + 1024;
  const cudaError_t e = cudaFuncSetAttribute(shared_attend_kernel<D, C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) { record_cuda_error("shared_attend attr", e); return PISA_ERR_CUDA; }
  const int grid = a.n_items < num_sms() ? a.n_items : num_sms();
  shared_attend_kernel<D, C><<<grid, kThreads, smem, s>>>(g, a, tm_q, tm_k, tm_v);
  return check_launch("shared_attend");
}

}  // namespace

size_t shared_attend_layout(const Geometry& g, char* ws, SharedPlan* p) {
  const int tpt = 128 / g.G;
  const size_t bh = (size_t)g.B * g.Hkv;
  p->threshold = share_threshold(g);
  p->span = g.C;
  p->words = (tpt + 31) / 32;
  p->tiles = (g.N + tpt - 1) / tpt;
  const int most = g.K * tpt / p->threshold + 1;                           // ... and leaf 0
  p->max_nodes = most < kSharedMax ? most : kSharedMax;
  const size_t tiles = bh * p->tiles;
  size_t o = 0;
  auto take = [&](size_t bytes) { char* r = ws + o; o += align_up(bytes, 256); return r; };
  p->node = (uint16_t*)take(tiles * p->max_nodes * 2);
  p->mask = (uint32_t*)take(tiles * p->max_nodes * p->words * 4);
  p->slot = nullptr;
  p->count = (int32_t*)take(tiles * 4);
  p->taken = (uint32_t*)take(bh * g.N * 4);
  p->chain = (int32_t*)take(tiles * 4);
  return o;
}

int launch_shared_attend(const Geometry& g, const void* q, const void* k, const void* v, const float* row_lse, float* o_acc,
                         const SharedPlan& plan, int32_t* ctr, int32_t* status, cudaStream_t s) {
  CUtensorMap tm_q, tm_k, tm_v;
  if (!qm_map_rows(&tm_q, q, g.d, g.Hq, g.N, g.B, g.qs, g.G, 128 / g.G) || !qm_map_rows(&tm_k, k, g.d, g.Hkv, g.N, g.B, g.ks, 1, g.C) ||
      !qm_map_rows(&tm_v, v, g.d, g.Hkv, g.N, g.B, g.vs, 1, g.C)) {
    record_cuda_error("shared_attend tensor maps", cudaErrorInvalidValue);
    return PISA_ERR_CUDA;
  }
  AttArgs a;
  a.plan = plan;
  a.row_lse = row_lse; a.o_acc = o_acc; a.ctr = ctr; a.status = status;
  a.q = (const __nv_bfloat16*)q; a.k = (const __nv_bfloat16*)k; a.v = (const __nv_bfloat16*)v;
  a.n_items = g.B * g.Hkv * plan.tiles;
  if (g.d == 128) return g.C == 128 ? launch_dc<128, 128>(g, a, tm_q, tm_k, tm_v, s) : launch_dc<128, 64>(g, a, tm_q, tm_k, tm_v, s);
  return g.C == 128 ? launch_dc<64, 128>(g, a, tm_q, tm_k, tm_v, s) : launch_dc<64, 64>(g, a, tm_q, tm_k, tm_v, s);
}

}  // namespace pisa
