// Masked dense attention over the selected leaves, query-major (see query_major.cuh; Eq. "selected sparse attention").
//
// Persistent, one CTA per SM.  A work item is NT 128-row tiles; warp 3 draws it from a global counter, ORs the tiles'
// selection bits into the list of steps (128 keys each) that some row needs, and hands item and list to the other roles
// through a two-deep ring.  Per step: K and V by TMA, S = Q K^T (tcgen05) -> P = exp(S - lse) in bf16 where the row
// selected the leaf, zero elsewhere (the row's denominator is known from the selection, so P is final), written over S in
// TMEM -> O += P V with P as the TMEM operand.  A warp none of whose rows selected a leaf skips its exponentials.  O is
// rounded and stored once per item: no accumulator in memory, no second pass.
// Roles: warp 0 TMA, warp 1 UMMA issuer, warp 2 idle, warp 3 scheduler, warps 4-11 and 12-19 two softmax / read-out
// groups, one per S / P buffer; inside a group two warps share a TMEM lane quarter, half of the columns each.  NT = 1: the
// buffers take alternate steps of the tile.  NT = 2: a buffer per tile, so that a step's keys and values (64 KB at d = 128)
// feed 256 rows.  The issuer walks the steps in order: the product with P that a buffer still owes, then the next S into
// it -- no barrier guards the buffer, the tensor pipe runs one thread's instructions in order.
// Measured at 8192 tokens, 16 KV heads, d = 128: P through shared memory with separate issuers took 2200 cycles per tile
// and step with NT = 1 and NT = 2 alike (each product waited for the other's queue).  An issuer per tile: 707 us against 653
// (4 x 4 KV heads, G = 4), 583 against 485 (C = 128) -- the pipe loses more by changing chains than one issuer's loop does,
// which is busy 1570 of 1855 cycles per tile and step, the chains' 1024 among them.
// Every wait is bounded.  What is not finite reaches only the rows that selected it (attend_row; finite inputs pay a test of
// the sums as they are read out).
#include "launch.cuh"
#include "lse_chunk.cuh"
#include "pisa_tensor.cuh"
#include "query_major.cuh"
#include "tc_utils.cuh"
#include "tma_map.cuh"

namespace pisa {

using namespace tc;

namespace {

constexpr int kAttThreads = 640;
constexpr int kMaxSteps = 256;                 // steps of one sequence: 32768 tokens
constexpr int kRing = 2;

template <bool V> struct Bool { static constexpr bool value = V; };

struct AttArgs {
  const float* row_lse;      // [Hq, len] per sequence, natural log
  const __nv_bfloat16 *q, *k, *v;   // for attend_row()
  __nv_bfloat16* out;        // strides of the geometry's `out`
  int two_terms;             // every sequence takes P in two bf16 terms (LO), not only those of one leaf
};

// One row over its own leaves only, by one warp.  The tiles multiply every value of a step with every row, zero weights
// included, so that a value (or a score) that is not finite reaches rows that did not select it or must not see it; rows that
// came out not finite are computed again here, where only what they selected takes part.
template <int D>
__device__ __forceinline__ void attend_row(const __nv_bfloat16* q, const __nv_bfloat16* k, long long ks, const __nv_bfloat16* v, long long vs,
                                           const uint32_t* bits, int t, int lgC, float sl2, float neg_lse2, bool round_p,
                                           __nv_bfloat16* out) {
  const int lane = threadIdx.x & 31;
  float acc[D / 32];
  bool gone = false;                             // every column is NaN, whatever follows
#pragma unroll
  for (int y = 0; y < D / 32; ++y) acc[y] = 0.f;
  for (int leaf = 0; leaf <= (t >> lgC) && !gone; ++leaf) {
    if (!((bits[leaf >> 5] >> (leaf & 31)) & 1u)) continue;
    const int end = min((leaf + 1) << lgC, t + 1);
    for (int j0 = leaf << lgC; j0 < end && !gone; j0 += 32) {
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
        p = ex2_approx(fmaf(s, sl2, neg_lse2));
        if (round_p) p = __bfloat162float(__float2bfloat16_rn(p));
      }
      for (int x = 0; x < min(32, end - j0); ++x) {
        const float px = __shfl_sync(0xffffffffu, p, x);
#pragma unroll
        for (int y = 0; y < D / 32; ++y) acc[y] = fmaf(px, __bfloat162float(v[(long long)(j0 + x) * vs + lane + 32 * y]), acc[y]);
      }
      bool nan = true;
#pragma unroll
      for (int y = 0; y < D / 32; ++y) nan = nan && acc[y] != acc[y];
      gone = __all_sync(0xffffffffu, nan);
    }
  }
#pragma unroll
  for (int y = 0; y < D / 32; ++y) out[lane + 32 * y] = __float2bfloat16_rn(acc[y]);
}

// K / V tiles in flight (one ring: K, V, K, V, ...): what two items' query tiles leave of 227 KB
__host__ __device__ constexpr int att_stages(int D, int NT) { return D == 128 ? (NT == 1 ? 5 : 3) : 8; }

// LO: P in two bf16 terms (an instantiation of its own: the registers would spill in the other) for sequences of one leaf, or
// for all of them (two_terms): shapes whose alternative is the exact fp32 path, which rounds no P, keep its precision.
template <int D, int C, int NT, bool LO>
__global__ void __launch_bounds__(kAttThreads, 1)
qm_attend_kernel(Geometry geo, qm::Args a, AttArgs at, const __grid_constant__ CUtensorMap tm_q,
                 const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = D / 64, SLAB = 128 * 128, TILE = KS * SLAB, NKV = att_stages(D, NT);
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;                        // [2][NT] query tiles of this item and the next
  uint8_t* sKV = sQ + 2 * NT * TILE;         // [NKV]
  __shared__ uint64_t q_full[2], q_empty[2], kv_full[NKV], kv_empty[NKV], s_full[2], p_full[2], o_full[2], o_empty[2],
      l_full[kRing], l_empty[kRing];
  __shared__ uint8_t s_list[kRing][kMaxSteps];
  __shared__ uint8_t s_need[NT == 2 ? kRing : 1][NT == 2 ? kMaxSteps : 1];   // NT = 2: which tiles need the step (bits 0, 1)
  __shared__ int4 s_item[kRing];             // (work item or -1, steps, steps of the first tile, of the second)
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  __shared__ volatile int s_again;           // some row came out not finite
  // this CTA's items: the last one + 1; the one before it stands in the score table (word `item`: nothing reads the scores any
  // more, and there are four of them at least for every item)
  __shared__ volatile int s_items;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1);
      mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 8);
      mbar_init(&o_full[i], 1); mbar_init(&o_empty[i], NT == 1 ? 16 : 8);
      mbar_init(&l_full[i], 1); mbar_init(&l_empty[i], 18);
    }
    for (int i = 0; i < NKV; ++i) { mbar_init(&kv_full[i], 1); mbar_init(&kv_empty[i], 1); }
    s_fail = 0;
    s_again = 0;
    s_items = 0;
    mbar_fence_init();
  }
  if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  grid_dependency();
  const uint32_t tmem = tmem_slot;           // S / P buffers at columns 0 / 128, O buffers at 256 / 384
  const int lgC = a.lgC, lgG = a.lgG, G = geo.G, tpt = 128 >> lgG;
  constexpr int LPS = 128 / C;               // leaves per step

  // the next ring entry: false when there is no more work (or something failed)
  auto next_item = [&](int it, int4& e) -> bool {
    const int r = it % kRing;
    if (!mbar_wait_bounded(&l_full[r], (uint32_t)((it / kRing) & 1))) { s_fail = 1; return false; }
    e = s_item[r];
    return e.x >= 0 && !s_fail;
  };
  auto done_item = [&](int it) {
    __syncwarp();
    if (lane == 0) mbar_arrive(&l_empty[it % kRing]);
  };
  auto needs = [&](int it, int j, int x) -> bool { return NT == 1 || ((s_need[NT == 2 ? it % kRing : 0][NT == 2 ? j : 0] >> x) & 1); };

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
      int n = 0, n0 = 0, n1 = 0;
      if (item < a.n_items) {
        const qm::Tile tl = qm::locate(geo, a, item, NT);
        const int W = (((tl.q.len + C - 1) >> lgC) + 31) >> 5, t0 = tl.tile * tpt * NT;
        const uint32_t* bits = a.bits + tl.q.bits_off + ((long long)tl.h * tl.q.len + t0) * W;
        const int nt = min(tpt * NT, tl.q.len - t0), na = min(tpt, nt);
        for (int w = 0; w < W && w * 32 <= ((t0 + nt - 1) >> lgC); ++w) {
          uint32_t v[2] = {0u, 0u};
          for (int k = lane; k < na; k += 32) v[0] |= bits[(long long)k * W + w];
          v[0] = __reduce_or_sync(0xffffffffu, v[0]);
          if (NT == 2) {
            for (int k = tpt + lane; k < nt; k += 32) v[1] |= bits[(long long)k * W + w];
            v[1] = __reduce_or_sync(0xffffffffu, v[1]);
          }
          const uint32_t mask = (1u << LPS) - 1u;
          const bool mine = lane < 32 / LPS;
          const bool on0 = mine && ((v[0] >> (lane * LPS)) & mask) != 0u, on1 = mine && ((v[1] >> (lane * LPS)) & mask) != 0u;
          const unsigned bal = __ballot_sync(0xffffffffu, on0 || on1);
          n0 += __popc(__ballot_sync(0xffffffffu, on0));
          n1 += __popc(__ballot_sync(0xffffffffu, on1));
          const int pos = n + __popc(bal & ((1u << lane) - 1u));
          if ((on0 || on1) && pos < kMaxSteps) {
            s_list[r][pos] = (uint8_t)(w * (32 / LPS) + lane);
            if (NT == 2) s_need[NT == 2 ? r : 0][NT == 2 ? pos : 0] = (uint8_t)((on0 ? 1 : 0) | (on1 ? 2 : 0));
          }
          n = min(n + __popc(bal), kMaxSteps);
        }
      }
      if (lane == 0) {
        s_item[r] = make_int4(item < a.n_items && ok ? item : -1, n, n0, n1);
        if (item < a.n_items) {
          reinterpret_cast<int*>(a.leaf)[item] = s_items;
          s_items = item + 1;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&l_full[r]);
      if (item >= a.n_items || !ok) break;
    }
  } else if (warp == 0) {
    // ------------------------------------------------ TMA producer
    int ld = 0;                                                    // tiles loaded into the ring so far
    int4 e;
    for (int it = 0; next_item(it, e); ++it) {
      const qm::Tile tl = qm::locate(geo, a, e.x, NT);
      if (lane == 0) {
        const int qb = it & 1;
        bool ok = it < 2 || mbar_wait_bounded(&q_empty[qb], (uint32_t)(((it >> 1) - 1) & 1));
        if (ok) {
          mbar_arrive_expect_tx(&q_full[qb], (uint32_t)(NT * TILE));
          for (int x = 0; x < NT; ++x)
            for (int ks = 0; ks < KS; ++ks)
              tma_load_4d(smem_u32(sQ + (qb * NT + x) * TILE + ks * SLAB), &tm_q, &q_full[qb], ks * 64, tl.h * G,
                          tl.q.tok + (tl.tile * NT + x) * tpt, tl.q.batch);
        }
        for (int j = 0; j < 2 * e.y && ok; ++j) {                  // K and V of every step
          const int n = ld + j, s = n % NKV, key = tl.q.tok + (int)s_list[it % kRing][j >> 1] * 128;
          ok = n < NKV || mbar_wait_bounded(&kv_empty[s], (uint32_t)((n / NKV - 1) & 1));
          if (!ok) break;
          mbar_arrive_expect_tx(&kv_full[s], (uint32_t)TILE);
          for (int ks = 0; ks < KS; ++ks)
            tma_load_4d(smem_u32(sKV + s * TILE + ks * SLAB), (j & 1) ? &tm_v : &tm_k, &kv_full[s], ks * 64, tl.h, key, tl.q.batch);
        }
        if (!ok) s_fail = 1;
      }
      ld += 2 * e.y;
      done_item(it);
    }
  } else if (warp == 1) {
    // ------------------------------------------------ UMMA issuer
    // The tensor pipe takes about 60 cycles per instruction from this warp; everything else in the loop is time it idles,
    // and the warp gets one issue slot in five.  So: counters instead of divisions, values that are the same in all lanes
    // made visibly so (shuffles), and no early exits -- after a wait that gave up the loop runs through without waiting
    // (its operands stay inside this CTA's memory) and the status word tells.
    const uint32_t idesc_s = make_idesc_bf16(128, 128, 0, 0);
    const uint32_t idesc_o = make_idesc_bf16(128, D, 0, 1);
    const uint32_t q_base = desc_lo(smem_u32(sQ), 0), k_base = desc_lo(smem_u32(sKV), 0), v_base = desc_lo(smem_u32(sKV), SLAB);
    bool dead = false;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (!dead && !mbar_try_wait(bar, parity) && !mbar_wait_bounded(bar, parity)) { dead = true; s_fail = 1; }
    };
    // what a buffer owes: the product of its P with the values of a step (stage < 0: nothing)
    struct Owed { int stage; uint32_t phase, p_phase, ob, o_wait; int rows; bool fresh, last, lo; };
    Owed owed[2];
    owed[0].stage = owed[1].stage = -1;
    uint32_t p_phase[2] = {0u, 0u}, o_count[2] = {0u, 0u};          // products per P buffer (parity); outputs per O buffer
    auto product = [&](const Owed& w, uint32_t sb) {
      wait(&p_full[sb], w.p_phase);
      wait(&kv_full[w.stage], w.phase);
      if (w.fresh && w.o_wait) wait(&o_empty[w.ob], w.o_wait & 1u);
      if (a.seqs != nullptr && w.rows < 128) {
        // packed: the rows past the sequence's end belong to its neighbour; their probabilities are zero, but a value
        // that is not finite would still reach the sum
        for (int x = lane; x < (128 - w.rows) * KS * 8; x += 32) {
          const int rr = w.rows + x / (KS * 8), ck = x % (KS * 8);
          st_shared_zero16(smem_u32(sKV + w.stage * TILE + (ck >> 3) * SLAB) + swz128(rr, ck & 7));
        }
        fence_proxy_async_smem();
        __syncwarp();
      }
      tcgen05_fence_after_sync();
      const uint32_t p0 = tmem + sb * 128u, d0 = tmem + 256u + w.ob * 128u, v0 = v_base + (uint32_t)(w.stage * (TILE >> 4));
      if (elect_one()) {
        if (!LO || !w.lo) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)                            // sixteen keys: eight columns of P, its halves 64 apart
            umma_bf16_ts(d0, p0 + (uint32_t)((kk >> 2) * 64 + (kk & 3) * 8), desc64(v0 + kk * (2048 >> 4)), idesc_o,
                         (!w.fresh || kk > 0) ? 1u : 0u);
        } else {
#pragma unroll 1
          for (int x = 0; x < 16; ++x) {                            // two terms of P
            const int kk = x >> 1;
            umma_bf16_ts(d0, p0 + (uint32_t)((kk >> 1) * 32 + (x & 1) * 16 + (kk & 1) * 8), desc64(v0 + (uint32_t)kk * (2048u >> 4)), idesc_o,
                         (!w.fresh || x > 0) ? 1u : 0u);
          }
        }
        if (w.last) umma_commit(&o_full[w.ob]);
      }
      __syncwarp();
    };
    auto release = [&](int stage) {
      if (elect_one()) umma_commit(&kv_empty[stage]);
      __syncwarp();
    };
    int st = 0, prev_v = -1;                                        // next ring stage; stage of the previous step's values
    uint32_t ph = 0u, par = 0u;                                     // its phase; parity of the step
    int4 e;
    for (int it = 0; next_item(it, e); ++it) {
      const int ny = __shfl_sync(0xffffffffu, e.y, 0), n0 = __shfl_sync(0xffffffffu, e.z, 0), n1 = __shfl_sync(0xffffffffu, e.w, 0);
      int len = 0x7fffffff;
      if (a.seqs != nullptr) len = qm::locate(geo, a, e.x, NT).q.len;
      const bool two_terms = at.two_terms || (a.seqs != nullptr ? len : geo.N) <= C;
      int seen[2] = {0, 0};
      wait(&q_full[it & 1], (uint32_t)((it >> 1) & 1));
      const uint32_t q_item = q_base + (uint32_t)((it & 1) * NT * (TILE >> 4));
      for (int j = 0; j < ny; ++j) {
        const int sk = st;
        const uint32_t phk = ph;
        if (++st == NKV) { st = 0; ph ^= 1u; }
        const int sv = st;
        const uint32_t phv = ph;
        if (++st == NKV) { st = 0; ph ^= 1u; }
        const int rows = (a.seqs != nullptr) ? len - (int)s_list[it % kRing][j] * 128 : 128;
        const uint32_t need = (NT == 2) ? __shfl_sync(0xffffffffu, (uint32_t)s_need[NT == 2 ? it % kRing : 0][NT == 2 ? j : 0], 0) : 1u;
#pragma unroll
        for (int x = 0; x < NT; ++x) {
          // NT = 1: owed[0] is the step before last, in this step's buffer; NT = 2: owed[x] is tile x's
          const uint32_t sb = (NT == 1) ? par : (uint32_t)x;
          if (owed[x].stage >= 0) {
            product(owed[x], sb);
            if (NT == 1) release(owed[x].stage);
            owed[x].stage = -1;
          }
          if (NT == 2 && x == 1 && prev_v >= 0) release(prev_v);    // both tiles' products of the previous step are out
          if (NT == 1) owed[0] = owed[1];
          if (!((need >> x) & 1u)) continue;
          wait(&kv_full[sk], phk);
          tcgen05_fence_after_sync();
          const uint32_t q0 = q_item + (uint32_t)(x * (TILE >> 4)), k0 = k_base + (uint32_t)(sk * (TILE >> 4));
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk) {
              const uint32_t o = (uint32_t)((kk >> 2) * SLAB + (kk & 3) * 32) >> 4;
              umma_bf16(tmem + sb * 128u, desc64(q0 + o), desc64(k0 + o), idesc_s, kk > 0);
            }
            umma_commit(&s_full[sb]);
          }
          __syncwarp();
          Owed& w = owed[NT == 1 ? 1 : x];
          w.stage = sv; w.phase = phv; w.rows = rows; w.lo = two_terms;
          const uint32_t pb = (NT == 1) ? par : (uint32_t)x;
          w.p_phase = (NT == 1) ? (p_phase[0] >> pb) & 1u : p_phase[x];
          if (NT == 1) p_phase[0] ^= 1u << pb; else p_phase[x] ^= 1u;
          w.ob = (NT == 1) ? (uint32_t)(it & 1) : (uint32_t)x;
          w.fresh = seen[x] == 0;
          if (w.fresh) {                                            // outputs of this buffer so far: 0 = nothing to wait for
            const uint32_t n = (NT == 1) ? (uint32_t)(it >> 1) : o_count[x]++;
            w.o_wait = n == 0u ? 0u : 2u | ((n - 1u) & 1u);
          }
          w.last = ++seen[x] == (x == 0 ? n0 : n1);
        }
        release(sk);
        if (NT == 2) prev_v = sv;
        par ^= 1u;
      }
      if (elect_one()) umma_commit(&q_empty[it & 1]);
      done_item(it);
    }
    // what is still owed, older steps first
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (owed[u].stage >= 0) product(owed[u], (NT == 1) ? par ^ (uint32_t)u : (uint32_t)u);
  } else if (warp >= 4) {
    // ------------------------------------------------ softmax and read-out
    const int grp = (warp - 4) >> 3, half = ((warp - 4) >> 2) & 1, quarter = warp & 3;
    const int row = quarter * 32 + lane, head = row & (G - 1);
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    const uint32_t s_base = tmem + lane_sel + (uint32_t)(grp * 128 + half * 64);   // this warp's columns of S, then of P
    const float sl2 = geo.scale * kLog2e;
    int kv = 0, cnt = 0, outs = 0;               // steps; steps of this group; outputs read by this group (NT = 2)
    int4 e;
    for (int it = 0; next_item(it, e); ++it) {
      const qm::Tile tl = qm::locate(geo, a, e.x, NT);
      const int t = (tl.tile * NT + (NT == 2 ? grp : 0)) * tpt + (row >> lgG), len = tl.q.len;
      const bool live = t < len;
      const int W = (((len + C - 1) >> lgC) + 31) >> 5;
      const uint32_t* bits = a.bits + tl.q.bits_off + ((long long)tl.h * len + (live ? t : 0)) * W;
      const uint8_t* list = s_list[it % kRing];
      float neg_lse2 = 0.f;
      if (live)
        neg_lse2 = -at.row_lse[(long long)geo.Hq * tl.q.cu + (long long)(tl.h * G + head) * len + t] * kLog2e;
      bool ok = true;
      constexpr int JS = (NT == 1) ? 2 : 1;
      int j = (NT == 1) ? ((kv ^ grp) & 1) : 0;   // this group's first step of the item
      uint32_t word = (live && j < e.y) ? bits[((int)list[j] * LPS) >> 5] : 0u;
      for (; j < e.y && ok; j += JS) {
        const int leaf0 = (int)list[j] * LPS, key0 = (int)list[j] * 128;
        const uint32_t mine = word >> (leaf0 & 31);
        if (live && j + JS < e.y) word = bits[((int)list[j + JS] * LPS) >> 5];      // in flight during this step
        if (!needs(it, j, grp)) continue;
        const int c = cnt++;
        const int vis = live ? t - key0 + 1 : 0;    // keys of the step this row may see
        ok = mbar_wait_bounded(&s_full[grp], (uint32_t)(c & 1));
        if (!ok) break;
        tcgen05_fence_after_sync();
        // (two bodies: a warp whose rows see all of their leaves -- nearly every one -- does without two instructions per key)
        const bool sel0 = live && ((mine >> ((half * 64) / C)) & 1u), sel1 = live && ((mine >> ((half * 64 + 32) / C)) & 1u);
        const int nv0 = sel0 ? max(0, min(32, vis - 64 * half)) : 0, nv1 = sel1 ? max(0, min(32, vis - 64 * half - 32)) : 0;
        auto probs = [&](int qq, bool sel, int nv, auto masked) {
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
              if (2 * x >= nv) p0 = 0.f;
              if (2 * x + 1 >= nv) p1 = 0.f;
            }
            const __nv_bfloat162 pp = __floats2bfloat162_rn(p0, p1);
            pk[x] = *reinterpret_cast<const uint32_t*>(&pp);
          }
          tmem_st_32x16(s_base + (uint32_t)(qq * 16), pk);                   // over columns of S this warp has already read
        };
        if (LO && (at.two_terms || len <= C)) {
          // P in two bf16 terms, sixteen columns each for 32 keys
#pragma unroll 1
          for (int qq = 0; qq < 2; ++qq) {
            uint32_t rr[32], pk[16];
            tmem_ld_32x32(s_base + (uint32_t)(qq * 32), rr);
            tmem_ld_wait();
#pragma unroll
            for (int part = 0; part < 2; ++part) {
#pragma unroll
              for (int x = 0; x < 16; ++x) {
                const int nv = qq ? nv1 : nv0;
                float p0 = 2 * x < nv ? ex2_approx(fmaf(__uint_as_float(rr[2 * x]), sl2, neg_lse2)) : 0.f;
                float p1 = 2 * x + 1 < nv ? ex2_approx(fmaf(__uint_as_float(rr[2 * x + 1]), sl2, neg_lse2)) : 0.f;
                __nv_bfloat162 pp = __floats2bfloat162_rn(p0, p1);
                if (part) pp = __floats2bfloat162_rn(p0 - __low2float(pp), p1 - __high2float(pp));
                pk[x] = *reinterpret_cast<const uint32_t*>(&pp);
              }
              tmem_st_32x16(s_base + (uint32_t)(qq * 32 + part * 16), pk);
            }
          }
        } else if (__any_sync(0xffffffffu, nv0 > 0 || nv1 > 0)) {
          if (__all_sync(0xffffffffu, (nv0 == 32 || !sel0) && (nv1 == 32 || !sel1))) {
            probs(0, sel0, nv0, Bool<false>());
            probs(1, sel1, nv1, Bool<false>());
          } else {
            probs(0, sel0, nv0, Bool<true>());
            probs(1, sel1, nv1, Bool<true>());
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
        if (lane == 0) mbar_arrive(&p_full[grp]);
      }
      kv += e.y;
      if (!ok) s_fail = 1;
      done_item(it);
      if (NT == 2 && (grp == 0 ? e.z : e.w) == 0) continue;                  // a pair without a second tile
      // read-out: this warp's share of the row's columns (NT = 1: both groups read the one tile)
      const int ob = (NT == 1) ? (it & 1) : grp;
      const uint32_t ph = (NT == 1) ? (uint32_t)((it >> 1) & 1) : (uint32_t)(outs & 1);
      ++outs;
      if (ok && !mbar_wait_bounded(&o_full[ob], ph)) { s_fail = 1; ok = false; }
      if (!ok) continue;                                                     // (next_item ends the loop on s_fail)
      tcgen05_fence_after_sync();
      constexpr int HC = (NT == 1) ? D / 4 : D / 2;
      const int col0 = ((NT == 1) ? grp * 2 + half : half) * HC;
      const uint32_t o_base = tmem + lane_sel + 256u + (uint32_t)(ob * 128 + col0);
      __nv_bfloat16* dst = at.out + (long long)tl.q.batch * geo.os[0] + (long long)(tl.q.tok + t) * geo.os[1] +
                           (long long)(tl.h * G + head) * geo.os[2] + col0;
      constexpr int LC = HC < 32 ? HC : 32;
      uint64_t finite[2] = {0ull, 0ull};                                     // NaN once a value is infinite or NaN
#pragma unroll
      for (int c0 = 0; c0 < HC; c0 += LC) {
        uint32_t rr[LC];
        if constexpr (LC == 32) tmem_ld_32x32(o_base + (uint32_t)c0, rr);
        else tmem_ld_32x16(o_base + (uint32_t)c0, rr);
        tmem_ld_wait();
        if (c0 + LC >= HC) {
          tcgen05_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&o_empty[ob]);
        }
#pragma unroll
        for (int x = 0; x < LC / 2; ++x)
          finite[x & 1] = fma2(pack2(__uint_as_float(rr[2 * x]), __uint_as_float(rr[2 * x + 1])), 0ull, finite[x & 1]);
        if (live)
#pragma unroll
          for (int q4 = 0; q4 < LC / 8; ++q4) {
            uint4 o;
            uint32_t* ow = &o.x;
#pragma unroll
            for (int x = 0; x < 4; ++x) {
              const __nv_bfloat162 pp = __floats2bfloat162_rn(__uint_as_float(rr[8 * q4 + 2 * x]), __uint_as_float(rr[8 * q4 + 2 * x + 1]));
              ow[x] = *reinterpret_cast<const uint32_t*>(&pp);
            }
            *reinterpret_cast<uint4*>(dst + c0 + 8 * q4) = o;
          }
      }
      float f0, f1;
      unpack2(add2(finite[0], finite[1]), f0, f1);
      if (live && f0 + f1 != 0.f) s_again = 1;
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.status, (int)PISA_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, 512);
  if (!s_again || s_fail) return;
  for (int item = s_items - 1; item >= 0; item = reinterpret_cast<const int*>(a.leaf)[item] - 1) {
    const qm::Tile tl = qm::locate(geo, a, item, NT);
    const int len = tl.q.len, W = (((len + C - 1) >> lgC) + 31) >> 5;
    const long long b = tl.q.batch, tok = tl.q.tok;
    for (int row = warp; row < 128 * NT; row += kAttThreads / 32) {
      const int t = tl.tile * NT * tpt + (row >> lgG), hq = tl.h * G + (row & (G - 1));
      if (t >= len) break;
      __nv_bfloat16* out = at.out + b * geo.os[0] + (tok + t) * geo.os[1] + hq * geo.os[2];
      float finite = 0.f;
#pragma unroll
      for (int y = 0; y < D / 32; ++y) finite = fmaf(__bfloat162float(out[lane + 32 * y]), 0.f, finite);
      if (!__any_sync(0xffffffffu, finite != finite)) continue;
      attend_row<D>(at.q + b * geo.qs[0] + (tok + t) * geo.qs[1] + hq * geo.qs[2], at.k + b * geo.ks[0] + tok * geo.ks[1] + tl.h * geo.ks[2],
                    geo.ks[1], at.v + b * geo.vs[0] + tok * geo.vs[1] + tl.h * geo.vs[2], geo.vs[1],
                    a.bits + tl.q.bits_off + ((long long)tl.h * len + t) * W, t, lgC, geo.scale * kLog2e,
                    -at.row_lse[(long long)geo.Hq * tl.q.cu + (long long)hq * len + t] * kLog2e, !(LO && (at.two_terms || len <= C)), out);
    }
  }
}

template <int D, int C, int NT, bool LO>
int launch_dcn(const Geometry& g, const qm::Args& a, const AttArgs& at, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
               const CUtensorMap& tm_v, cudaStream_t s) {
  const size_t smem = (size_t)(D / 64) * (2 * NT + att_stages(D, NT)) * 128 * 128 + 1024;
  const int grid = a.n_items < num_sms() ? a.n_items : num_sms();
  return launch_dependent<qm_attend_kernel<D, C, NT, LO>>("qm_attend", dim3((unsigned)grid), kAttThreads, smem, s, g, a, at, tm_q, tm_k, tm_v);
}
template <int D, int C>
int launch_dc(const Geometry& g, const qm::Args& a, const AttArgs& at, const CUtensorMap& tm_q, const CUtensorMap& tm_k,
              const CUtensorMap& tm_v, bool lo, cudaStream_t s) {
  if (lo) return a.tiles == 2 ? launch_dcn<D, C, 2, true>(g, a, at, tm_q, tm_k, tm_v, s) : launch_dcn<D, C, 1, true>(g, a, at, tm_q, tm_k, tm_v, s);
  return a.tiles == 2 ? launch_dcn<D, C, 2, false>(g, a, at, tm_q, tm_k, tm_v, s) : launch_dcn<D, C, 1, false>(g, a, at, tm_q, tm_k, tm_v, s);
}

}  // namespace

int launch_qm_attend(const Geometry& g, const qm::Args& a, const void* q, const void* k, const void* v, long long tokens,
                     const float* row_lse, void* out, bool one_leaf, bool two_terms, cudaStream_t s) {
  CUtensorMap tm_q, tm_k, tm_v;
  if (!qm_map_rows(&tm_q, q, g.d, g.Hq, tokens, g.B, g.qs, g.G, 128 / g.G) ||
      !qm_map_rows(&tm_k, k, g.d, g.Hkv, tokens, g.B, g.ks, 1, 128) ||
      !qm_map_rows(&tm_v, v, g.d, g.Hkv, tokens, g.B, g.vs, 1, 128)) {
    record_cuda_error("qm_attend tensor maps", cudaErrorInvalidValue);
    return PISA_ERR_CUDA;
  }
  AttArgs at;
  at.two_terms = two_terms;
  one_leaf |= two_terms;
  at.row_lse = row_lse; at.out = (__nv_bfloat16*)out;
  at.q = (const __nv_bfloat16*)q; at.k = (const __nv_bfloat16*)k; at.v = (const __nv_bfloat16*)v;
  if (g.d == 128) return g.C == 128 ? launch_dc<128, 128>(g, a, at, tm_q, tm_k, tm_v, one_leaf, s) : launch_dc<128, 64>(g, a, at, tm_q, tm_k, tm_v, one_leaf, s);
  return g.C == 128 ? launch_dc<64, 128>(g, a, at, tm_q, tm_k, tm_v, one_leaf, s) : launch_dc<64, 64>(g, a, at, tm_q, tm_k, tm_v, one_leaf, s);
}

}  // namespace pisa
