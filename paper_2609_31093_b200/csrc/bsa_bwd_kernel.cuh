// Backward of the block-sparse attention with the selected indices held fixed (App. B), d = 128 or 64.
// Included by tensor_path.cu inside its unnamed namespace: it works on the same inverted
// (key block -> tokens) lists and work items as the forward attention kernel.
//
// A tile is 64 gathered rows (64 / G tokens) against one key block; scores and their gradients are held transposed, a TMEM lane
// per key, so that P and dS are operands of the key and value gradients where they lie:
//   S^T = K Q^T,  dP^T = V dO^T                                            (UMMA, 128 x 64)
//   P = 2^(S*scale*log2e - lse2),  dS = P o (dP - delta) * scale           (TMEM -> bf16: both over S^T in TMEM, dS also to
//                                                                           shared memory)
//   dV += P^T dO,  dK += dS^T Q      (A from TMEM; kept there over all tiles of a work item, then added to fp32 in memory)
//   dQ^T = K^T dS^T                  (-> fp32 accumulator by vector reductions, heads innermost)
// Warps: 8 gather the Q and dO rows (cp.async, three pairs of tiles in flight), one loads an item's K and V, one draws items and
// lays out tiles ahead of everybody, one issues the products, 8 do the element-wise step and the dV / dK read-out, 4 reduce dQ.
// TMEM: dV at columns 0..127, dK at 128.., two buffers of 128 from 256 on: S, over which P and dS are written, and dP, whose
// columns are free once both are there and take dQ.  The next tile's S and dP go out before this tile's other products, so that
// its element-wise step runs under them, as do the gathers and the reductions (32 KB a tile, 16 bytes per clock and SM at best).
// C = 64: the upper 64 key rows are zero (so are their scores and gradients) and never read out; d = 64: the rows are one
// 64-column slab, and the upper lanes of dQ^T, fed from the neighbouring slab, are not read out.
// Measured: 32768 tokens, 32 heads, C = 128, K = 32: 7.0 ms, 570 TFLOP/s of the five products (one CTA that walked a tile of 128
// rows with all its warps in step: 12.3 ms); with C = 64, K = 16 1.9 ms (3.1 ms).  What bounds it: the issuing warp's chain, about
// 3700 cycles a tile of which the tensor pipe works 1660.
// delta = rowsum(dO o O) comes from a small kernel of its own or from the dense way's preparation.
// What is not finite reaches only what it belongs to: where a row sees a part of its own block only, the products multiply the
// rest by zero.  So keys that are not finite count as zero and their scores as NaN, and so do, in tiles with rows of the block's
// own leaf, rows whose denominator or delta shows that they are not finite.
#pragma once

constexpr int kBwdThreads = 736;
constexpr int kBwdRows = 64;           // rows of a tile
constexpr int kBwdStages = 3;          // pairs of Q / dO tiles
constexpr int kBwdRing = 8;            // tiles the scheduler may run ahead

struct BwdArgs {
  const __nv_bfloat16* q;
  const __nv_bfloat16* k;
  const __nv_bfloat16* v;
  const __nv_bfloat16* dout;      // [B, N, Hq, D], strides of `out`
  const float* lse;               // [B, Hq, N] natural log
  const float* delta;             // [B, Hq, N]
  const float2* stat;             // or, instead of both: [B, Hkv, N, G] (-lse * log2 e, -delta), from the dense path's preparation
  const int32_t* entry_off;
  const int32_t* item_off;
  const int32_t* item_key;
  const int32_t* entries;
  int nkeys, Mk, NW;
  float* dq_acc;                  // [B, Hkv, N, D, G] fp32
  float* dk_acc;                  // [B, N, Hkv, D] fp32
  float* dv_acc;
  int32_t* work_ctr;              // next work item (zero on entry)
  int kv_tma;                     // keys and values through the tensor maps
  int32_t* status;
  Gate gate;
};

// delta[b, hq, t] = sum_d dO[b,t,hq,d] * O[b,t,hq,d]; one warp per row
__global__ void __launch_bounds__(256) bwd_delta_kernel(Geometry geo, const __nv_bfloat16* __restrict__ out,
                                                        const __nv_bfloat16* __restrict__ dout,
                                                        float* __restrict__ delta) {
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  const long long rows = (long long)geo.B * geo.N * geo.Hq;
  if (w >= rows) return;
  const int hq = (int)(w % geo.Hq);
  const long long bt = w / geo.Hq;
  const int t = (int)(bt % geo.N), b = (int)(bt / geo.N);
  const long long off = (long long)b * geo.os[0] + (long long)t * geo.os[1] + (long long)hq * geo.os[2];
  float s = 0.f;
  for (int dd = lane; dd < geo.d; dd += 32) s += __bfloat162float(out[off + dd]) * __bfloat162float(dout[off + dd]);
  s = warp_sum(s);
  if (lane == 0) delta[((long long)b * geo.Hq + hq) * geo.N + t] = s;
}

// fp32 -> bf16, contiguous
// fp32 accumulator rows of `row2` element pairs, dense -> bf16 rows `dst_pitch2` pairs apart (a chunk of
// KV heads writes its columns of the caller's [B, N, Hkv, d] tensor)
__global__ void __launch_bounds__(256) bwd_convert_kernel(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst,
                                                          long long n2, int row2, long long dst_pitch2, Gate gate) {
  if (gate.off_list()) return;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n2) return;
  const float2 x = reinterpret_cast<const float2*>(src)[i];
  const long long row = i / row2;
  reinterpret_cast<__nv_bfloat162*>(dst)[row * dst_pitch2 + (i - row * row2)] = __floats2bfloat162_rn(x.x, x.y);
}

__device__ __forceinline__ ItemInfo item_info_keys(const int32_t* item_key, const int32_t* item_off,
                                                   const int32_t* entry_off, int item, int tpt) {
  ItemInfo r;
  r.key = item_key[item];
  const int local = item - item_off[r.key];
  const int list0 = entry_off[r.key], cnt = entry_off[r.key + 1] - list0;
  const int tiles = (cnt + tpt - 1) / tpt;
  const int first = local * kItemTiles;
  r.ntiles = min(kItemTiles, tiles - first);
  r.e_begin = list0 + first * tpt;
  r.e_end = list0 + cnt;
  return r;
}

template <bool V> struct BwdOwn { static constexpr bool value = V; };

template <int C, int D, bool WIDE>
__global__ void __launch_bounds__(kBwdThreads, 1) bsa_bwd_kernel(Geometry geo, BwdArgs a, const __grid_constant__ CUtensorMap tm_k,
                                                                 const __grid_constant__ CUtensorMap tm_v) {
  if (a.gate.off_list()) return;
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = D / 64, CH = D / 8;                    // 64-column slabs, 16-byte chunks of a row
  constexpr int R_SLAB = kBwdRows * 128, R_TILE = KS * R_SLAB, KV_SLAB = 128 * 128, KV_TILE = KS * KV_SLAB, DS_TILE = 128 * 128;
  constexpr int NS = kBwdStages, R = kBwdRing;
  uint8_t* smem = align1024(smem_raw);
  uint8_t* sK = smem;
  uint8_t* sV = sK + KV_TILE;                               // (right behind K: d = 64 reads past K's only slab)
  uint8_t* sdS = sV + KV_TILE;                              // [2]
  uint8_t* sQ = sdS + 2 * DS_TILE;                          // [NS]
  uint8_t* sdO = sQ + NS * R_TILE;                          // [NS]
  __shared__ uint64_t m_full[R], m_empty[R], qd_full[NS], qd_empty[NS], kv_full, kv_empty, k_seen, s_full[2], e_done[2], dq_full[2], dq_empty[2],
      acc_full, acc_empty;
  __shared__ int s_ent[R][kBwdRows];                        // a tile's entries (token | slot << 24, -1 = none)
  __shared__ int4 s_tkey[R];                                // its (unit, leaf, flags: 1 / 2 = first / last of its item, 4 = own-leaf rows)
  __shared__ __align__(16) float2 s_stat[NS][kBwdRows];     // per row (-lse * log2 e, -delta); (-inf, 0) where there is no row
  __shared__ float s_kscale[128];                           // per key scale * log2 e, NaN where the key is not finite
  __shared__ volatile int s_total;                          // number of tiles of this CTA, known once the walk has ended
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < R; ++i) { mbar_init(&m_full[i], 1); mbar_init(&m_empty[i], 22); }
    for (int i = 0; i < NS; ++i) { mbar_init(&qd_full[i], 256); mbar_init(&qd_empty[i], 1); }
    mbar_init(&kv_full, 1); mbar_init(&kv_empty, 1); mbar_init(&k_seen, C / 32);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_full[i], 1); mbar_init(&e_done[i], 8);
      mbar_init(&dq_full[i], 1); mbar_init(&dq_empty[i], 4);
    }
    mbar_init(&acc_full, 1); mbar_init(&acc_empty, 8);
    s_total = 0x7fffffff;
    s_fail = 0;
    mbar_fence_init();
  }
  if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
  if (C == 64)                                              // key rows beyond the block: zero for good
    for (int i = tid; i < 2 * KS * 64 * 8; i += kBwdThreads) {
      const int slab = i / (64 * 8), x = i - slab * (64 * 8);
      st_shared_zero16(smem_u32(sK + slab * KV_SLAB) + 64 * 128 + x * 16);
    }
  fence_proxy_async_smem();
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  constexpr uint32_t T_DV = 0u, T_DK = 128u, T_BUF = 256u;         // buffer b at T_BUF + 128 b: S (then P, dS), dP (then dQ) 64 further

  const int G = geo.G, lgG = 31 - __clz(G), tpt = kBwdRows >> lgG;
  const float sl2 = geo.scale * kLog2e;
  // a tile's ring entry, or false when the walk has ended before it (every role walks the CTA's tiles; bounded as in lse_ws_kernel)
  auto wait_tile = [&](int it) -> bool {
    for (uint32_t i = 0; i < (1u << 24); ++i) {
      if (mbar_try_wait(&m_full[it % R], (uint32_t)((it / R) & 1))) return true;
      if (it >= s_total || s_fail) return false;
    }
    s_fail = 1;
    return false;
  };
  auto done_tile = [&](int it) {
    __syncwarp();
    if (lane == 0) mbar_arrive(&m_empty[it % R]);
  };
  // (code size: with all roles' loops unrolled 62 % of the instruction fetches hit the SM's cache, and more stalls were for
  // instructions than for anything else: 8.4 ms at 32768 tokens, 32 heads, C = 128, now 7.0)

  if (warp < 8) {
    // ------------------------------------------------ gather: a tile's Q and dO rows and their statistics
    constexpr int RPP = 256 / CH;                           // rows per pass
    const int ck = tid % CH, rb = tid / CH;
    for (int it = 0; wait_tile(it); ++it) {
      const int st = it % NS, mr = it % R;
      if (it >= NS && !mbar_wait_bounded(&qd_empty[st], (uint32_t)((it / NS - 1) & 1))) { s_fail = 1; break; }
      const int bh = s_tkey[mr].x, b = bh / geo.Hkv, h = bh % geo.Hkv;
      const int* ents = s_ent[mr];
      const __nv_bfloat16* qb = a.q + (long long)b * geo.qs[0] + (long long)(h * G) * geo.qs[2] + ck * 8;
      const __nv_bfloat16* ob = a.dout + (long long)b * geo.os[0] + (long long)(h * G) * geo.os[2] + ck * 8;
      const uint32_t off = (uint32_t)(st * R_TILE + (ck >> 3) * R_SLAB);
      const uint32_t dq0 = smem_u32(sQ) + off, do0 = smem_u32(sdO) + off;
#pragma unroll 1
      for (int row = rb; row < kBwdRows; row += RPP) {
        const int ent = ents[row >> lgG];
        const uint32_t d = swz128(row, ck & 7);
        if (ent >= 0) {
          cp_async16(dq0 + d, qb + (long long)(ent & 0xFFFFFF) * geo.qs[1] + (long long)(row & (G - 1)) * geo.qs[2]);
          cp_async16(do0 + d, ob + (long long)(ent & 0xFFFFFF) * geo.os[1] + (long long)(row & (G - 1)) * geo.os[2]);
        } else {
          st_shared_zero16(dq0 + d);
          st_shared_zero16(do0 + d);
        }
      }
      if (tid < kBwdRows) {
        const int ent = ents[tid >> lgG];
        float2 x = make_float2(-CUDART_INF_F, 0.f);
        if (ent >= 0) {
          const int t = ent & 0xFFFFFF, head = tid & (G - 1);
          if (a.stat != nullptr) {
            x = a.stat[((long long)bh * geo.N + t) * G + head];
          } else {
            const long long li = ((long long)b * geo.Hq + h * G + head) * geo.N + t;
            x = make_float2(-a.lse[li] * kLog2e, -a.delta[li]);
          }
        }
        s_stat[st][tid] = x;
      }
      fence_proxy_async_smem();                             // zero-filled rows (plain stores) -> async proxy
      cp_async_arrive_noinc(&qd_full[st]);                  // fires when this thread's copies have landed
      done_tile(it);
    }
    cp_async_wait_all();
  } else if (warp == 8) {
    // ------------------------------------------------ an item's keys and values
    int n_item = 0;
    for (int it = 0; wait_tile(it); ++it) {
      const int4 key = s_tkey[it % R];
      if (key.z & 1) {
        if (n_item >= 1 && !mbar_wait_bounded(&kv_empty, (uint32_t)((n_item - 1) & 1))) { s_fail = 1; break; }
        ++n_item;
        const int b = key.x / geo.Hkv, h = key.x % geo.Hkv;
        if (a.kv_tma) {                                     // (own memory, no multicast; rows past N read as zero)
          if (lane == 0) {
            mbar_arrive_expect_tx(&kv_full, (uint32_t)(2 * KS * C * 128));
            for (int ks = 0; ks < KS; ++ks) {
              tma_load_4d(smem_u32(sK + ks * KV_SLAB), &tm_k, &kv_full, ks * 64, h, key.y * C, b);
              tma_load_4d(smem_u32(sV + ks * KV_SLAB), &tm_v, &kv_full, ks * 64, h, key.y * C, b);
            }
          }
        } else {                                            // strides a tensor map cannot hold
          const int ck = lane % CH;
          const __nv_bfloat16* kb = a.k + (long long)b * geo.ks[0] + (long long)h * geo.ks[2] + ck * 8;
          const __nv_bfloat16* vb = a.v + (long long)b * geo.vs[0] + (long long)h * geo.vs[2] + ck * 8;
          const uint32_t k0 = smem_u32(sK + (ck >> 3) * KV_SLAB), v0 = smem_u32(sV + (ck >> 3) * KV_SLAB);
#pragma unroll 1
          for (int row = lane / CH; row < C; row += 32 / CH) {
            const long long t = (long long)key.y * C + row;
            const uint32_t d = swz128(row, ck & 7);
            if (t < geo.N) {
              cp_async16(k0 + d, kb + t * geo.ks[1]);
              cp_async16(v0 + d, vb + t * geo.vs[1]);
            } else {
              st_shared_zero16(k0 + d);
              st_shared_zero16(v0 + d);
            }
          }
          cp_async_wait_all();
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(&kv_full);
        }
      }
      done_tile(it);
    }
  } else if (warp == 9) {
    // ------------------------------------------------ scheduler: draws work items, lays out their tiles
    const int n_items = a.item_off[a.nkeys], tpt128 = 128 >> lgG;
    int it = 0;
    bool ok = true;
    while (ok) {
      int item = 0;
      if (lane == 0) item = atomicAdd(a.work_ctr, 1);
      item = __shfl_sync(0xffffffffu, item, 0);
      if (item >= n_items) break;
      const ItemInfo inf = item_info_keys(a.item_key, a.item_off, a.entry_off, item, tpt128);
      const int bh = inf.key / (a.NW * a.Mk), leaf = inf.key % a.Mk;
      const int e_end = min(inf.e_end, inf.e_begin + inf.ntiles * tpt128), n = (e_end - inf.e_begin + tpt - 1) / tpt;
      auto fetch = [&](int j, int x) -> int {               // the tile's entry x
        const int e = inf.e_begin + j * tpt + x;
        return (j < n && x < tpt && e < e_end) ? a.entries[e] : -1;
      };
      int nx0 = fetch(0, lane), nx1 = fetch(0, lane + 32);
      for (int j = 0; j < n && ok; ++j, ++it) {
        const int e0 = nx0, e1 = nx1, mr = it % R;
        nx0 = fetch(j + 1, lane);
        nx1 = fetch(j + 1, lane + 32);
        if (it >= R) ok = mbar_wait_bounded(&m_empty[mr], (uint32_t)((it / R - 1) & 1));
        ok = __all_sync(0xffffffffu, ok && !s_fail);
        if (!ok) break;
        s_ent[mr][lane] = e0;
        s_ent[mr][lane + 32] = e1;
        const bool own = __any_sync(0xffffffffu, (e0 >= 0 && (e0 & 0xFFFFFF) / C == leaf) || (e1 >= 0 && (e1 & 0xFFFFFF) / C == leaf));
        if (lane == 0) s_tkey[mr] = make_int4(bh, leaf, (j == 0 ? 1 : 0) | (j == n - 1 ? 2 : 0) | (own ? 4 : 0), 0);
        __syncwarp();
        if (lane == 0) mbar_arrive(&m_full[mr]);            // release: the ring entry is complete
      }
    }
    if (!ok) s_fail = 1;
    if (lane == 0) s_total = it;
  } else if (warp == 10) {
    // ------------------------------------------------ UMMA issuer (after a wait that gave up it runs through without waiting)
    // The warp stands still while the pipe works, and the pipe while the warp does anything else: what the next run of
    // instructions waits for is looked at before the last ones of this run.
    const uint32_t idesc_s = make_idesc_bf16(128, kBwdRows, 0, 0);   // keys x rows, both K-major over d
    const uint32_t idesc_g = make_idesc_bf16(128, D, 0, 1);          // keys (TMEM) x d, over the rows
    const uint32_t idesc_q = make_idesc_bf16(128, kBwdRows, 1, 1);   // d x rows, over the keys
    const uint32_t k0 = desc_lo(smem_u32(sK), 0), v0 = desc_lo(smem_u32(sV), 0), kt0 = desc_lo(smem_u32(sK), KV_SLAB);
    const uint32_t q_base = desc_lo(smem_u32(sQ), 0), o_base = desc_lo(smem_u32(sdO), 0), ds_base = desc_lo(smem_u32(sdS), DS_TILE);
    constexpr uint32_t R_LBO = (uint32_t)(R_SLAB >> 4) << 16;        // the row tiles as MN-major operands
    constexpr int HOLD = 2;                                 // instructions still to go out when the next run is looked at
    bool dead = false;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      if (!dead && !mbar_try_wait(bar, parity) && !mbar_wait_bounded(bar, parity)) { dead = true; s_fail = 1; }
    };
    int n_item = 0, it = 0;                                 // items begun; the tile whose S and dP are next
    uint32_t st = 0u, st_ph = 0u, st_prev = 0u;             // its stage and phase; stage of the tile before
    uint32_t flags = 0u, prev = 0u;                         // its flags; those of the tile before, whose gradients are owed (8: there is one)
    bool known = false, rows_ready = false, e_ready = false;
    // gradients of tile it - 1 once its P and dS are there: dQ^T first, so that the reducers have it by the time the tile after
    // next wants its columns.  look: see to tile it + 1 meanwhile
    auto gradients = [&](bool look) {
      const uint32_t buf = (uint32_t)((it - 1) & 1);
      if ((prev & 1u) && n_item >= 2) wait(&acc_empty, (uint32_t)((n_item - 2) & 1));
      if (!e_ready) wait(&e_done[buf], (uint32_t)(((it - 1) >> 1) & 1));
      e_ready = false;
      tcgen05_fence_after_sync();
      const uint32_t off = st_prev * (uint32_t)(R_TILE >> 4);
      const uint32_t qm = q_base + R_LBO + off, om = o_base + R_LBO + off, s0 = ds_base + buf * (uint32_t)(DS_TILE >> 4);
      const uint32_t tb = tmem + T_BUF + buf * 128u, acc = (prev & 1u) ? 0u : 1u;
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < C / 16; ++kk)
          umma_bf16(tb + 64u, desc64(kt0 + kk * (2048 >> 4)), desc64(s0 + kk * (2048 >> 4)), idesc_q, kk > 0);
        umma_commit(&dq_full[buf]);
#pragma unroll
        for (int kk = 0; kk < kBwdRows / 16; ++kk)
          umma_bf16_ts(tmem + T_DV, tb + (uint32_t)(kk * 16), desc64(om + kk * (2048 >> 4)), idesc_g, kk > 0 ? 1u : acc);
#pragma unroll
        for (int kk = 0; kk < kBwdRows / 16 - HOLD; ++kk)
          umma_bf16_ts(tmem + T_DK, tb + (uint32_t)(kk * 16 + 8), desc64(qm + kk * (2048 >> 4)), idesc_g, kk > 0 ? 1u : acc);
      }
      __syncwarp();
      if (look) {
        const int nx = it + 1;
        const uint32_t ns = (st + 1u == (uint32_t)NS) ? 0u : st + 1u;
        const bool m = mbar_test(&m_full[nx % R], (uint32_t)((nx / R) & 1)), r = mbar_test(&qd_full[ns], st_ph ^ (ns == 0u ? 1u : 0u));
        const uint32_t word = (m ? 256u : 0u) | (r ? 512u : 0u) | ((uint32_t)s_tkey[nx % R].z & 7u);   // (no such tile yet: whatever stands there)
        const uint32_t w0 = __shfl_sync(0xffffffffu, word, 0);
        known = (w0 & 256u) != 0u;
        rows_ready = known && (w0 & 512u) != 0u;
        flags = w0 & 255u;
      }
      if (elect_one()) {
#pragma unroll
        for (int kk = kBwdRows / 16 - HOLD; kk < kBwdRows / 16; ++kk)
          umma_bf16_ts(tmem + T_DK, tb + (uint32_t)(kk * 16 + 8), desc64(qm + kk * (2048 >> 4)), idesc_g, kk > 0 ? 1u : acc);
        umma_commit(&qd_empty[st_prev]);
        if (prev & 2u) {
          umma_commit(&acc_full);
          umma_commit(&kv_empty);
        }
      }
      __syncwarp();
    };
    for (;; ++it) {
      if (!known) {
        if (!wait_tile(it)) break;
        flags = (uint32_t)__shfl_sync(0xffffffffu, s_tkey[it % R].z, 0);
      }
      known = false;
      if (flags & 1u) {
        if (prev & 8u) {                                    // the keys of the item before go with its last gradients
          gradients(false);
          prev = 0u;
        }
        wait(&k_seen, (uint32_t)(n_item & 1));
        ++n_item;
      }
      const uint32_t buf = (uint32_t)(it & 1), own = flags;
      if (!rows_ready) wait(&qd_full[st], st_ph);
      rows_ready = false;
      if (own & 4u) {                                       // rows that are not finite (see the head of this file)
#pragma unroll 1
        for (int r0 = 0; r0 < kBwdRows; r0 += 32) {
          const float2 x = s_stat[st][r0 + lane];
          const bool bad = !(fabsf(x.y) < CUDART_INF_F) || !(x.x < CUDART_INF_F);
          if (bad) s_stat[st][r0 + lane].x = CUDART_NAN_F;
          for (unsigned m = __ballot_sync(0xffffffffu, bad); m != 0u; m &= m - 1u) {
            const int row = r0 + __ffs(m) - 1;
            if (lane < KS * 8) {
              const uint32_t d = st * (uint32_t)R_TILE + (uint32_t)((lane >> 3) * R_SLAB) + swz128(row, lane & 7);
              st_shared_zero16(smem_u32(sQ) + d);
              st_shared_zero16(smem_u32(sdO) + d);
            }
          }
        }
        __syncwarp();
      }
      fence_proxy_async_smem();
      tcgen05_fence_after_sync();
      const uint32_t q0 = q_base + st * (uint32_t)(R_TILE >> 4), o0 = o_base + st * (uint32_t)(R_TILE >> 4), tb = tmem + T_BUF + buf * 128u;
      auto mma_s = [&](int kk, uint32_t d, uint32_t a0, uint32_t b0) {
        const uint32_t ko = (uint32_t)((kk >> 2) * KV_SLAB + (kk & 3) * 32) >> 4, ro = (uint32_t)((kk >> 2) * R_SLAB + (kk & 3) * 32) >> 4;
        umma_bf16(d, desc64(a0 + ko), desc64(b0 + ro), idesc_s, kk > 0);
      };
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) mma_s(kk, tb, k0, q0);
      }
      __syncwarp();
      done_tile(it);
      if (it >= 2) wait(&dq_empty[buf], (uint32_t)(((it >> 1) - 1) & 1));    // dP goes where the dQ^T of the tile before last was
      tcgen05_fence_after_sync();
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < D / 16 - HOLD; ++kk) mma_s(kk, tb + 64u, v0, o0);
      }
      __syncwarp();
      if (prev & 8u) e_ready = __all_sync(0xffffffffu, mbar_test(&e_done[buf ^ 1u], (uint32_t)(((it - 1) >> 1) & 1)));
      if (elect_one()) {
#pragma unroll
        for (int kk = D / 16 - HOLD; kk < D / 16; ++kk) mma_s(kk, tb + 64u, v0, o0);
        umma_commit(&s_full[buf]);
      }
      __syncwarp();
      if (prev & 8u) gradients(true);
      prev = own | 8u;
      st_prev = st;
      if (++st == (uint32_t)NS) { st = 0u; st_ph ^= 1u; }
    }
    if (prev & 8u) gradients(false);
  } else if (warp >= 11 && warp < 19) {
    // ------------------------------------------------ element-wise step (lane = key), dV / dK read-out
    const int quarter = warp & 3, half = (warp - 11) >> 2;            // TMEM lane quarter; half of the tile's rows
    const int key = quarter * 32 + lane;
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    const bool active = quarter * 32 < C;                             // C = 64: the upper lanes stay zero
    int n_item = 0;
    for (int it = 0; wait_tile(it); ++it) {
      const int4 tk = s_tkey[it % R];
      const float4* stat = reinterpret_cast<const float4*>(s_stat[it % NS] + half * 32);
      uint8_t* ds = sdS + (it & 1) * DS_TILE;
      if ((tk.z & 1) && half == 0 && active) {
        // the item's keys: one that is not finite counts as zero (see the head of this file)
        if (!mbar_wait_bounded(&kv_full, (uint32_t)(n_item & 1))) { s_fail = 1; break; }
        const uint32_t k_row = smem_u32(sK);
        float f = 0.f;
#pragma unroll 4
        for (int ck = 0; ck < CH; ++ck) {
          const uint32_t d = k_row + (uint32_t)((ck >> 3) * KV_SLAB) + swz128(key, ck & 7);
          uint32_t w[4];
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(d));
#pragma unroll
          for (int x = 0; x < 4; ++x) f = fmaf(__uint_as_float(w[x] << 16), 0.f, fmaf(__uint_as_float(w[x] & 0xFFFF0000u), 0.f, f));
        }
        if (f != 0.f) {                                               // (0 or NaN)
#pragma unroll 1
          for (int ck = 0; ck < CH; ++ck) st_shared_zero16(k_row + (uint32_t)((ck >> 3) * KV_SLAB) + swz128(key, ck & 7));
        }
        s_kscale[key] = f != 0.f ? CUDART_NAN_F : sl2;
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&k_seen);
      }
      // (s_full says that the rows had landed; their statistics were written by then)
      if (!mbar_wait_bounded(&qd_full[it % NS], (uint32_t)((it / NS) & 1)) ||
          !mbar_wait_bounded(&s_full[it & 1], (uint32_t)((it >> 1) & 1))) { s_fail = 1; break; }
      tcgen05_fence_after_sync();
      if (active) {
        // sixteen rows at a time, P and dS over their own columns of S (two bodies: a branch inside would cut the unrolled
        // chains into blocks that wait for one another, 3000 cycles a tile)
        const float ks = s_kscale[key];
        auto step = [&](auto own) {
#pragma unroll 1
          for (int cc = 0; cc < 2; ++cc) {
            const uint32_t s_base = tmem + lane_sel + T_BUF + (uint32_t)((it & 1) * 128 + half * 32 + cc * 16);
            uint32_t rs[16], rp[16], pk[8], dk[8];
            tmem_ld_32x16(s_base, rs);
            tmem_ld_32x16(s_base + 64u, rp);
            tmem_ld_wait();
#pragma unroll
            for (int jx = 0; jx < 8; ++jx) {
              const float4 x = stat[cc * 8 + jx];                     // two rows
              float p0 = ex2_approx(fmaf(__uint_as_float(rs[2 * jx]), ks, x.x));
              float p1 = ex2_approx(fmaf(__uint_as_float(rs[2 * jx + 1]), ks, x.z));
              float d0 = p0 * (__uint_as_float(rp[2 * jx]) + x.y) * geo.scale;
              float d1 = p1 * (__uint_as_float(rp[2 * jx + 1]) + x.w) * geo.scale;
              if (own.value) {                                        // rows of the block's own leaf see keys up to themselves
                const int r = half * 32 + cc * 16 + 2 * jx, j = tk.y * C + key;
                const int e0 = s_ent[it % R][r >> lgG], e1 = s_ent[it % R][(r + 1) >> lgG];
                const bool off0 = e0 < 0 || j > (e0 & 0xFFFFFF), off1 = e1 < 0 || j > (e1 & 0xFFFFFF);
                p0 = off0 ? 0.f : p0; d0 = off0 ? 0.f : d0;
                p1 = off1 ? 0.f : p1; d1 = off1 ? 0.f : d1;
              }
              const __nv_bfloat162 pp = __floats2bfloat162_rn(p0, p1), dd = __floats2bfloat162_rn(d0, d1);
              pk[jx] = *reinterpret_cast<const uint32_t*>(&pp);
              dk[jx] = *reinterpret_cast<const uint32_t*>(&dd);
            }
            tmem_st_32x8(s_base, pk);
            tmem_st_32x8(s_base + 8u, dk);
#pragma unroll
            for (int q = 0; q < 2; ++q)
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(smem_u32(ds) + swz128(key, half * 4 + cc * 2 + q)), "r"(dk[4 * q]),
                           "r"(dk[4 * q + 1]), "r"(dk[4 * q + 2]), "r"(dk[4 * q + 3])
                           : "memory");
          }
        };
        if (tk.z & 4) step(BwdOwn<true>());
        else step(BwdOwn<false>());
        tmem_st_wait();
        fence_proxy_async_smem();
      }
      tcgen05_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&e_done[it & 1]);
      done_tile(it);
      if (tk.z & 2) {
        // the item's dV (half 0) or dK (half 1): lane = key, TMEM column = d
        if (!mbar_wait_bounded(&acc_full, (uint32_t)(n_item & 1))) { s_fail = 1; break; }
        ++n_item;
        tcgen05_fence_after_sync();
        const int b = tk.x / geo.Hkv, h = tk.x % geo.Hkv;
        const long long t = (long long)tk.y * C + key;
        float* dst = (half == 0 ? a.dv_acc : a.dk_acc) + (((long long)b * geo.N + t) * geo.Hkv + h) * D;
        if (active) {
#pragma unroll 1
          for (int c0 = 0; c0 < D; c0 += 16) {
            uint32_t r[16];
            tmem_ld_32x16(tmem + lane_sel + (half == 0 ? T_DV : T_DK) + (uint32_t)c0, r);
            tmem_ld_wait();
            if (t < geo.N)
#pragma unroll
              for (int q4 = 0; q4 < 4; ++q4)
                asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + c0 + 4 * q4),
                             "f"(__uint_as_float(r[4 * q4])), "f"(__uint_as_float(r[4 * q4 + 1])),
                             "f"(__uint_as_float(r[4 * q4 + 2])), "f"(__uint_as_float(r[4 * q4 + 3]))
                             : "memory");
          }
        }
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty);
      }
    }
  } else if (warp >= 19) {
    // ------------------------------------------------ reducer: dQ^T (lane = column d, TMEM column = tile row) -> fp32 accumulator
    const int quarter = warp & 3, row = quarter * 32 + lane;
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    for (int it = 0; wait_tile(it); ++it) {
      const int buf = it & 1, bh = s_tkey[it % R].x;
      const int* ents = s_ent[it % R];
      float* acc_d = a.dq_acc + (long long)bh * geo.N * (long long)(D * G) + (long long)row * G;
      const uint32_t tok_bytes = (uint32_t)(D * G * 4);
      if (!mbar_wait_bounded(&dq_full[buf], (uint32_t)((it >> 1) & 1))) { s_fail = 1; break; }
      tcgen05_fence_after_sync();
      if (quarter * 32 < D) {                               // lanes beyond d hold nothing of use
        uint32_t ra[32], rb[32];                            // all of them at once: dP of the tile after next waits for the columns
        tmem_ld_32x32(tmem + lane_sel + T_BUF + (uint32_t)(buf * 128 + 64), ra);
        tmem_ld_32x32(tmem + lane_sel + T_BUF + (uint32_t)(buf * 128 + 96), rb);
        tmem_ld_wait();
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&dq_empty[buf]);
        auto at = [&](int e) { return reinterpret_cast<float*>(reinterpret_cast<char*>(acc_d) + (uint64_t)(uint32_t)(e & 0xFFFFFF) * tok_bytes); };
        reduce_columns<WIDE>(ra, G, lane, [&](int r) { return ents[r >> lgG]; }, at);
        reduce_columns<WIDE>(rb, G, lane, [&](int r) { return ents[(32 + r) >> lgG]; }, at);
      } else if (lane == 0) {
        mbar_arrive(&dq_empty[buf]);
      }
      done_tile(it);
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.status, (int)PISA_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, 512);
}
