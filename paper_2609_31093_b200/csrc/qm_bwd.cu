// The dense masked backward's kernels (see qm_bwd.cuh).
#include "launch.cuh"
#include "lse_chunk.cuh"
#include "pisa_tensor.cuh"
#include "qm_bwd.cuh"
#include "step_ring.cuh"
#include "tc_utils.cuh"
#include "tma_map.cuh"

namespace pisa {

using namespace tc;
using qmb::Args;

namespace {

// ------------------------------------------------------------------ preparation

// One block per 128-row tile.  Bound by reading out and dout once (16-byte loads, D / 8 lanes per row).
template <int D>
__global__ void __launch_bounds__(256) qm_bwd_prep_kernel(Geometry geo, Args a) {
  extern __shared__ uint32_t s_bits[];                      // [tokens][W], then [W] their union
  grid_dependency();
  if (blockIdx.x == 0 && threadIdx.x < 2) a.ctr[threadIdx.x] = 0;
  const int G = geo.G, lgG = a.lgG, tpt = 128 >> lgG, K = geo.K;
  const qmb::Loc loc = qmb::locate<qmb::kTiles>(geo, a, blockIdx.x);
  const int len = loc.q.len, h = loc.h, t0 = loc.part * tpt, nt = min(tpt, len - t0);
  const int M1 = (len + geo.C - 1) >> a.lgC, W = (M1 + 31) >> 5, tiles = (len + tpt - 1) / tpt;
  for (int i = threadIdx.x; i < (tpt + 1) * W; i += blockDim.x) s_bits[i] = 0u;
  constexpr int LPR = D / 8, RPP = 256 / LPR;               // lanes per row, rows per pass
  const int sub = threadIdx.x % LPR;
  const long long base = (long long)loc.q.batch * geo.os[0] + (long long)loc.q.tok * geo.os[1] + (long long)(h * G) * geo.os[2] + sub * 8;
#pragma unroll 4
  for (int r = threadIdx.x / LPR; r < 128; r += RPP) {
    const int t = t0 + (r >> lgG), hd = r & (G - 1);
    float s = 0.f;
    if (t < len) {
      float x[8], y[8];
      const long long o = base + (long long)t * geo.os[1] + (long long)hd * geo.os[2];
      Elem<__nv_bfloat16>::load_chunk(a.out + o, x);
      Elem<__nv_bfloat16>::load_chunk(a.dout + o, y);
#pragma unroll
      for (int e = 0; e < 8; ++e) s = fmaf(x[e], y[e], s);
    }
#pragma unroll
    for (int o = LPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (sub == 0 && t < len) {
      const float l = a.lse[(long long)geo.Hq * loc.q.cu + (long long)(h * G + hd) * len + t];
      a.stat[loc.q.leaf_off + ((long long)h * len + t) * G + hd] = make_float2(l == -CUDART_INF_F ? l : l < CUDART_INF_F ? -l * kLog2e : CUDART_NAN_F, -s);
    }
  }
  __syncthreads();
  const int32_t* idx = a.idx + (long long)geo.Hkv * K * loc.q.cu + ((long long)h * len + t0) * K;
  for (int i = threadIdx.x; i < nt * K; i += blockDim.x) {
    const int k = i / K, leaf = idx[i], c = (t0 + k) >> a.lgC;
    if (leaf >= 0 && leaf <= c) atomicOr(&s_bits[k * W + (leaf >> 5)], 1u << (leaf & 31));
    else if ((geo.debug & PISA_DEBUG_BOUNDS) && leaf != -1) atomicExch(a.status, (int)PISA_ERR_BOUNDS);
  }
  __syncthreads();
  uint32_t* bits = a.bits + loc.q.bits_off + ((long long)h * len + t0) * W;
  for (int i = threadIdx.x; i < nt * W; i += blockDim.x) {
    bits[i] = s_bits[i];
    if (s_bits[i] != 0u) atomicOr(&s_bits[tpt * W + i % W], s_bits[i]);
  }
  __syncthreads();
  for (int k = threadIdx.x; k < nt; k += blockDim.x) {      // a row without blocks counts for nothing, whatever it holds
    uint32_t any = 0u;
    for (int w = 0; w < W; ++w) any |= s_bits[k * W + w];
    for (int hd = 0; hd < G && any == 0u; ++hd)
      a.stat[loc.q.leaf_off + ((long long)h * len + t0 + k) * G + hd] = make_float2(-CUDART_INF_F, 0.f);
  }
  uint32_t* tb = a.tbits + loc.q.up_off + (long long)h * tiles * W + loc.part;
  int steps = 0;                                            // 128-key blocks the tile needs
  for (int w = threadIdx.x; w < W; w += blockDim.x) {
    const uint32_t u = s_bits[tpt * W + w];
    tb[(long long)w * tiles] = u;
    steps += geo.C == 128 ? __popc(u) : __popc((u | (u >> 1)) & 0x55555555u);
  }
  if (a.count != nullptr && steps > 0) atomicAdd(a.count, (uint32_t)steps);
}

// ------------------------------------------------------------------ shared by the two product kernels
//
// A scheduler warp draws items and lays out their steps in a ring (step_ring.cuh); every other role walks steps.  Roles:
// warp 0 TMA producer, warp 1 UMMA issuer, warp 2 row metadata (kv kernel), warp 3 scheduler, warps 4-19 two groups of eight
// (TMEM lane quarter = warp % 4) that turn the first two products into the operands of the next ones.  Every wait is
// bounded; after one that gave up the roles run through without waiting and the status word tells.
constexpr int kBwdThreads2 = 640;

template <bool V> struct Bool { static constexpr bool value = V; };
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&p);
}
__device__ __forceinline__ bool all_finite(const uint32_t (&r)[32]) {
  uint64_t s[2] = {0ull, 0ull};                             // NaN once a value is infinite or NaN
#pragma unroll
  for (int x = 0; x < 16; ++x) s[x & 1] = fma2(pack2(__uint_as_float(r[2 * x]), __uint_as_float(r[2 * x + 1])), 0ull, s[x & 1]);
  float a, b;
  unpack2(add2(s[0], s[1]), a, b);
  return a + b == 0.f;
}
// N floats of a row -> bf16, 16 bytes at a time
template <int N>
__device__ __forceinline__ void store_row(__nv_bfloat16* dst, const uint32_t (&r)[N]) {
#pragma unroll
  for (int q4 = 0; q4 < N / 8; ++q4) {
    uint4 o;
    uint32_t* ow = &o.x;
#pragma unroll
    for (int x = 0; x < 4; ++x) ow[x] = pack_bf16(__uint_as_float(r[8 * q4 + 2 * x]), __uint_as_float(r[8 * q4 + 2 * x + 1]));
    *reinterpret_cast<uint4*>(dst + 8 * q4) = o;
  }
}
// Two probabilities and their dS: p = 2^(s * sl2 + bias), d = p * (dp * scale - delta * scale).  The logit scale belongs in
// front of the rounding to bf16, not behind the sums: the roundings are then those of the list-driven kernel, and where the
// terms of a sum cancel (a key of large norm with most of a row's probability) they are what the result's error is made of.
// Packed arithmetic: seven instructions for two elements.
__device__ __forceinline__ void prob_grad2(uint32_t s0, uint32_t s1, uint32_t dp0, uint32_t dp1, uint64_t sl2, uint64_t bias, uint64_t sc, uint64_t ndelta,
                                           float& p0, float& p1, float& d0, float& d1) {
  float z0, z1;
  unpack2(fma2(pack2(__uint_as_float(s0), __uint_as_float(s1)), sl2, bias), z0, z1);
  p0 = ex2_approx(z0);
  p1 = ex2_approx(z1);
  unpack2(mul2(pack2(p0, p1), fma2(pack2(__uint_as_float(dp0), __uint_as_float(dp1)), sc, ndelta)), d0, d1);
}
// rows [first, rows) of `slabs` swizzled 64-column slabs become zero (one warp)
__device__ __forceinline__ void zero_rows(uint8_t* base, int slab_bytes, int slabs, int first, int rows) {
  const int lane = threadIdx.x & 31;
  for (int x = lane; x < (rows - first) * slabs * 8; x += 32) {
    const int r = first + x / (slabs * 8), ck = x % (slabs * 8);
    st_shared_zero16(smem_u32(base + (ck >> 3) * slab_bytes) + swz128(r, ck & 7));
  }
}

// ------------------------------------------------------------------ dK, dV

// TMEM: S^T halves (64 query rows each) at columns 0 / 64, dP^T at 128 / 192, dV at 256, dK at 384.  The two halves of a
// step are a double buffer: while one is turned into P^T and dS^T, the tensor pipe works on the other.
// Floor per step (128 rows x 128 keys): 2.6 K cycles of the tensor pipe (an N = 64 chain is bound by re-reading A from
// shared memory), 64 KB of Q and dO from L2 (3 K cycles at the 22 bytes per clock an SM gets); measured 3.8 K.
template <int D, int C>
__global__ void __launch_bounds__(kBwdThreads2, 1)
qm_bwd_kv_kernel(Geometry geo, Args a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_do,
                 const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = D / 64, SLAB = 128 * 128, TILE = KS * SLAB, NS = (D == 128) ? 2 : 4, LPS = 128 / C;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sK = smem;
  uint8_t* sV = sK + TILE;
  uint8_t* sQ = sV + TILE;                    // [NS] (Q, dO)
  __shared__ StepRing ring;
  __shared__ uint64_t st_full[NS], st_empty[NS], meta_full[NS], kv_full, kv_empty, s_full[2], p_full[2], acc_full, acc_empty;
  __shared__ __align__(16) float s_bias[NS][LPS][128], s_delta[NS][128];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  grid_dependency();
  if (a.gate.off_dense()) return;
  if (tid == 0) {
    ring_init(ring, 19);
    for (int i = 0; i < NS; ++i) { mbar_init(&st_full[i], 1); mbar_init(&st_empty[i], 1); mbar_init(&meta_full[i], 1); }
    mbar_init(&kv_full, 1); mbar_init(&kv_empty, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 8); }
    mbar_init(&acc_full, 1); mbar_init(&acc_empty, 16);
    s_fail = 0;
    mbar_fence_init();
  }
  if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  const int G = geo.G, lgG = a.lgG, tpt = 128 >> lgG, lgC = a.lgC;
  bool dead = false;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!dead && !mbar_try_wait(bar, parity) && !mbar_wait_bounded(bar, parity)) { dead = true; s_fail = 1; }
  };
  int n = 0;                                                  // ring position
  int4 e;

  if (warp == 3) {
    // ------------------------------------------------ scheduler
    for (bool ok = true; ok;) {
      int item = 0;
      if (lane == 0) item = atomicAdd(a.ctr, 1);
      item = __shfl_sync(0xffffffffu, item, 0);
      if (item >= a.n_keys) { ring_push(ring, n, make_int4(0, 0, kEnd, 0), &s_fail); break; }
      const qmb::Loc loc = qmb::locate<qmb::kKeys>(geo, a, item);
      const int len = loc.q.len, W = (((len + C - 1) >> lgC) + 31) >> 5, tiles = (len + tpt - 1) / tpt;
      const int leaf0 = loc.part * LPS, first = (loc.part * 128) / tpt;
      const uint32_t* tb = a.tbits + loc.q.up_off + ((long long)loc.h * W + (leaf0 >> 5)) * tiles;
      const int sp = loc.part == 0 ? a.splits0 : a.splits;
      int held = -1, flags = kFirst;                          // the last step found so far: pushed once the next one is known
      for (int base = first + loc.split; base < tiles && ok; base += 128 * sp) {
        unsigned m4[4];                                       // 128 tiles per round trip
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const int t = base + (32 * x + lane) * sp;
          m4[x] = t < tiles ? tb[t] >> (leaf0 & 31) : 0u;
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
          for (unsigned m = __ballot_sync(0xffffffffu, (m4[x] & ((1u << LPS) - 1u)) != 0u); m != 0u && ok; m &= m - 1u) {
            if (held >= 0) { ok = ring_push(ring, n, make_int4(item, held, flags, 0), &s_fail); flags = 0; }
            held = base + (32 * x + __ffs(m) - 1) * sp;
          }
      }
      if (ok) ok = ring_push(ring, n, held >= 0 ? make_int4(item, held, flags | kLast, 0) : make_int4(item, 0, kFirst | kLast | kEmpty, 0), &s_fail);
    }
  } else if (warp == 0) {
    // ------------------------------------------------ TMA producer
    int items = 0, step = 0;
    qmb::Loc loc;
    while (ring_pop(ring, n, e, &s_fail)) {
      if (e.z & kEmpty) continue;
      if (e.z & kFirst) {
        loc = qmb::locate<qmb::kKeys>(geo, a, e.x);
        if (items > 0) wait(&kv_empty, (uint32_t)((items - 1) & 1));
        if (lane == 0 && !dead) {
          mbar_arrive_expect_tx(&kv_full, (uint32_t)(2 * TILE));
          for (int ks = 0; ks < KS; ++ks) {
            tma_load_4d(smem_u32(sK + ks * SLAB), &tm_k, &kv_full, ks * 64, loc.h, loc.q.tok + loc.part * 128, loc.q.batch);
            tma_load_4d(smem_u32(sV + ks * SLAB), &tm_v, &kv_full, ks * 64, loc.h, loc.q.tok + loc.part * 128, loc.q.batch);
          }
        }
        ++items;
      }
      const int s = step % NS;
      if (step >= NS) wait(&st_empty[s], (uint32_t)((step / NS - 1) & 1));
      if (lane == 0 && !dead) {
        mbar_arrive_expect_tx(&st_full[s], (uint32_t)(2 * TILE));
        for (int ks = 0; ks < KS; ++ks) {
          tma_load_4d(smem_u32(sQ + 2 * s * TILE + ks * SLAB), &tm_q, &st_full[s], ks * 64, loc.h * G, loc.q.tok + e.y * tpt, loc.q.batch);
          tma_load_4d(smem_u32(sQ + (2 * s + 1) * TILE + ks * SLAB), &tm_do, &st_full[s], ks * 64, loc.h * G, loc.q.tok + e.y * tpt, loc.q.batch);
        }
      }
      __syncwarp();
      ++step;
    }
  } else if (warp == 2) {
    // ------------------------------------------------ row metadata: -lse2 where the row selected the leaf, -delta
    int step = 0;
    qmb::Loc loc;
    while (ring_pop(ring, n, e, &s_fail)) {
      if (e.z & kEmpty) continue;
      if (e.z & kFirst) loc = qmb::locate<qmb::kKeys>(geo, a, e.x);
      const int s = step % NS, len = loc.q.len, W = (((len + C - 1) >> lgC) + 31) >> 5, leaf0 = loc.part * LPS, t0 = e.y * tpt;
      const long long row0 = (long long)loc.h * len + t0;
      float2 st[4];
      uint32_t wd[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int r = lane + 32 * x, t = t0 + (r >> lgG);
        st[x] = make_float2(-CUDART_INF_F, 0.f);
        wd[x] = 0u;
        if (t < len) {
          st[x] = a.stat[loc.q.leaf_off + row0 * G + r];
          wd[x] = a.bits[loc.q.bits_off + (row0 + (r >> lgG)) * W + (leaf0 >> 5)] >> (leaf0 & 31);
        }
      }
      if (step >= NS) wait(&st_empty[s], (uint32_t)((step / NS - 1) & 1));
      // Rows that must not be multiplied as they are: those that count for nothing (past the sequence's end, where a packed
      // neighbour's lie, or without blocks), and those that hold something not finite (their denominator is NaN or their
      // delta not finite), unless only their dO does and they selected and see all of the step's keys
      uint32_t off[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int r = lane + 32 * x;
        constexpr uint32_t all = (1u << LPS) - 1u;
        const bool none = st[x].x == -CUDART_INF_F, nan = st[x].x != st[x].x;
        const bool whole = (wd[x] & all) == all && t0 + (r >> lgG) >= loc.part * 128 + 127;
        const bool bad = none || nan || (!whole && !(fabsf(st[x].y) < CUDART_INF_F));
        off[x] = __ballot_sync(0xffffffffu, bad);
#pragma unroll
        for (int lf = 0; lf < LPS; ++lf) s_bias[s][lf][r] = ((wd[x] >> lf) & 1u) ? (bad && !none ? CUDART_NAN_F : st[x].x) : -CUDART_INF_F;
        s_delta[s][r] = bad ? 0.f : st[x].y * geo.scale;
      }
      if ((off[0] | off[1] | off[2] | off[3]) != 0u) {
        wait(&st_full[s], (uint32_t)((step / NS) & 1));
#pragma unroll
        for (int x = 0; x < 4; ++x)
          for (uint32_t m = off[x]; m != 0u; m &= m - 1u) {
            const int r = 32 * x + __ffs(m) - 1;
            if (lane < 16 * KS)                             // eight chunks of 16 bytes per 64 columns, Q and dO
              st_shared_zero16(smem_u32(sQ + (2 * s + lane / (8 * KS)) * TILE + ((lane >> 3) % KS) * SLAB) + swz128(r, lane & 7));
          }
        fence_proxy_async_smem();
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&meta_full[s]);
      ++step;
    }
  } else if (warp == 1) {
    // ------------------------------------------------ UMMA issuer
    const uint32_t idesc_s = make_idesc_bf16(128, 64, 0, 0), idesc_g = make_idesc_bf16(128, D, 0, 1);
    const uint32_t k0 = desc_lo(smem_u32(sK), 0), v0 = desc_lo(smem_u32(sV), 0);
    const uint32_t q_s = desc_lo(smem_u32(sQ), 0), q_g = desc_lo(smem_u32(sQ), SLAB);
    int step = 0, items = 0, prev = -1, prev_flags = 0;       // prev: stage of the step whose second half is still owed
    // S^T and dP^T of one half of the step in `stage`
    auto scores = [&](uint32_t half, int stage) {
      tcgen05_fence_after_sync();
      const uint32_t b = (uint32_t)(2 * stage * (TILE >> 4)) + half * (8192u >> 4);
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t o = (uint32_t)((kk >> 2) * SLAB + (kk & 3) * 32) >> 4;
          umma_bf16(tmem + half * 64u, desc64(k0 + o), desc64(q_s + b + o), idesc_s, kk > 0);
        }
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk) {
          const uint32_t o = (uint32_t)((kk >> 2) * SLAB + (kk & 3) * 32) >> 4;
          umma_bf16(tmem + 128u + half * 64u, desc64(v0 + o), desc64(q_s + b + (TILE >> 4) + o), idesc_s, kk > 0);
        }
        umma_commit(&s_full[half]);
      }
      __syncwarp();
    };
    // dV += P^T dO, dK += dS^T Q of that half; parity: the step's
    auto grads = [&](uint32_t half, int stage, uint32_t parity, bool fresh) {
      wait(&p_full[half], parity);
      tcgen05_fence_after_sync();
      const uint32_t b = q_g + (uint32_t)(2 * stage * (TILE >> 4)) + half * (8192u >> 4);
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)                        // sixteen rows: eight columns, the two warps' parts 32 apart
          umma_bf16_ts(tmem + 256u, tmem + half * 64u + (uint32_t)((kk >> 1) * 32 + (kk & 1) * 8),
                       desc64(b + (TILE >> 4) + kk * (2048 >> 4)), idesc_g, (!fresh || kk > 0) ? 1u : 0u);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          umma_bf16_ts(tmem + 384u, tmem + 128u + half * 64u + (uint32_t)((kk >> 1) * 32 + (kk & 1) * 8),
                       desc64(b + kk * (2048 >> 4)), idesc_g, (!fresh || kk > 0) ? 1u : 0u);
      }
      __syncwarp();
    };
    auto owed = [&]() {
      grads(1u, prev, (uint32_t)((step - 1) & 1), false);
      if (elect_one()) {
        umma_commit(&st_empty[prev]);
        if (prev_flags & kLast) umma_commit(&acc_full);
      }
      __syncwarp();
    };
    while (ring_pop(ring, n, e, &s_fail)) {
      if (e.z & kEmpty) {                                     // (the read-out of the item before must not wait for a later step)
        if (prev >= 0) owed();
        prev = -1;
        continue;
      }
      const int s = step % NS;
      if (e.z & kFirst) wait(&kv_full, (uint32_t)(items & 1));
      wait(&st_full[s], (uint32_t)((step / NS) & 1));
      wait(&meta_full[s], (uint32_t)((step / NS) & 1));       // (rows that count for nothing are zero)
      scores(0u, s);
      if (prev >= 0) owed();
      scores(1u, s);
      if ((e.z & kLast) && elect_one()) umma_commit(&kv_empty);
      __syncwarp();
      if ((e.z & kFirst) && items > 0) wait(&acc_empty, (uint32_t)((items - 1) & 1));
      grads(0u, s, (uint32_t)(step & 1), (e.z & kFirst) != 0);
      prev = s; prev_flags = e.z;
      if (e.z & kFirst) ++items;
      ++step;
    }
    if (prev >= 0) owed();
  } else {
    // ------------------------------------------------ P^T, dS^T and the read-out
    const int grp = (warp - 4) >> 3, part = ((warp - 4) >> 2) & 1, quarter = warp & 3;
    const int row = quarter * 32 + lane;                      // key of the item
    const int lf = (LPS == 2) ? row >> 6 : 0;
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    const int col0 = grp * 64 + part * 32;                    // first of this warp's query rows
    const uint32_t base = tmem + lane_sel + (uint32_t)col0;
    const uint64_t sl2 = pack2(geo.scale * kLog2e, geo.scale * kLog2e), sc = pack2(geo.scale, geo.scale);
    int step = 0, items = 0;
    qmb::Loc loc;
    while (ring_pop(ring, n, e, &s_fail)) {
      if (e.z & kFirst) loc = qmb::locate<qmb::kKeys>(geo, a, e.x);
      const int key = loc.part * 128 + row;
      if (!(e.z & kEmpty)) {
        const int s = step % NS;
        const float* bias = s_bias[s][lf] + col0;
        const float* delta = s_delta[s] + col0;
        wait(&meta_full[s], (uint32_t)((step / NS) & 1));
        // rows of this warp's columns whose token is not before the warp's last key need the causal comparison
        const int tok0 = e.y * tpt + (col0 >> lgG);
        const bool diag = tok0 < loc.part * 128 + quarter * 32 + 31;
        const bool any = __any_sync(0xffffffffu, bias[lane] != -CUDART_INF_F) &&
                         (e.y * tpt + ((col0 + 31) >> lgG) >= loc.part * 128 + quarter * 32);
        wait(&s_full[grp], (uint32_t)(step & 1));
        tcgen05_fence_after_sync();
        uint32_t pk[16], dk[16];
        if (any) {
          uint32_t rs[32], rp[32];
          tmem_ld_32x32(base, rs);
          tmem_ld_32x32(base + 128u, rp);
          tmem_ld_wait();
          auto run = [&](auto masked) {
#pragma unroll
            for (int x = 0; x < 16; ++x) {
              const float2 bi = *reinterpret_cast<const float2*>(bias + 2 * x), de = *reinterpret_cast<const float2*>(delta + 2 * x);
              float p0, p1, d0, d1;
              prob_grad2(rs[2 * x], rs[2 * x + 1], rp[2 * x], rp[2 * x + 1], sl2, pack2(bi.x, bi.y), sc, pack2(de.x, de.y), p0, p1, d0, d1);
              if (masked.value) {
                if (e.y * tpt + ((col0 + 2 * x) >> lgG) < key) p0 = d0 = 0.f;
                if (e.y * tpt + ((col0 + 2 * x + 1) >> lgG) < key) p1 = d1 = 0.f;
              }
              pk[x] = pack_bf16(p0, p1);
              dk[x] = pack_bf16(d0, d1);
            }
          };
          if (diag) run(Bool<true>()); else run(Bool<false>());
        } else {
#pragma unroll
          for (int x = 0; x < 16; ++x) pk[x] = dk[x] = 0u;
        }
        tmem_st_32x16(base, pk);                              // over columns this warp has already read
        tmem_st_32x16(base + 128u, dk);
        tmem_st_wait();
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[grp]);
        ++step;
      }
      if (!(e.z & kLast)) continue;
      // read-out: [dV | dK], a quarter of the columns per warp that shares the lanes
      constexpr int CPW = 2 * D / 4;
      const int w4 = (warp - 4) >> 2, which = (w4 * CPW) / D, c0 = w4 * CPW - which * D;
      const bool live = key < loc.q.len;
      const long long orow = ((loc.q.cu + key) * geo.Hkv + loc.h) * D + c0;
      const bool direct = (loc.part == 0 ? a.splits0 : a.splits) == 1;
      // does a row of this item select the key?  (asked only for sums that are not finite)
      auto selected = [&]() -> bool {
        const int len = loc.q.len, W = (((len + C - 1) >> lgC) + 31) >> 5, leaf = key >> lgC, sp = loc.part == 0 ? a.splits0 : a.splits;
        for (int tile = (loc.part * 128) / tpt + loc.split; tile * tpt < len; tile += sp)
          for (int t = max(key, tile * tpt); t < min(len, (tile + 1) * tpt); ++t)
            if ((a.bits[loc.q.bits_off + ((long long)loc.h * len + t) * W + (leaf >> 5)] >> (leaf & 31)) & 1u) return true;
        return false;
      };
      if (e.z & kEmpty) {
        if (direct && live) {
          __nv_bfloat16* dst = (which ? a.dk : a.dv) + orow;
#pragma unroll
          for (int x = 0; x < CPW; x += 8) *reinterpret_cast<uint4*>(dst + x) = make_uint4(0u, 0u, 0u, 0u);
        }
        continue;
      }
      wait(&acc_full, (uint32_t)(items & 1));
      tcgen05_fence_after_sync();
#pragma unroll
      for (int x = 0; x < CPW; x += 32) {
        uint32_t r[32];
        tmem_ld_32x32(tmem + lane_sel + 256u + (uint32_t)(which * 128 + c0 + x), r);
        tmem_ld_wait();
        if (x + 32 >= CPW) {
          tcgen05_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty);
        }
        if (!live) continue;
        if (!all_finite(r) && !selected()) {
#pragma unroll
          for (int y = 0; y < 32; ++y) r[y] = 0u;
        }
        if (direct) {
          store_row<32>((which ? a.dk : a.dv) + orow + x, r);
        } else {
          const long long arow = a.splits > 1 ? orow : (((long long)loc.q.pyr_row * geo.Hkv + loc.h) * 128 + row) * D + c0;
          float* dst = (which ? a.dk_acc : a.dv_acc) + arow + x;
#pragma unroll
          for (int y = 0; y < 32; y += 4)
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + y), "f"(__uint_as_float(r[y])),
                         "f"(__uint_as_float(r[y + 1])), "f"(__uint_as_float(r[y + 2])), "f"(__uint_as_float(r[y + 3]))
                         : "memory");
        }
      }
      ++items;
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.status, (int)PISA_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------ dQ

// One row of dQ over its own leaves only, by one warp (as attend_row in qm_attend.cu)
template <int D>
__device__ __forceinline__ void dq_row(const __nv_bfloat16* q, const __nv_bfloat16* dout, const __nv_bfloat16* k, long long ks,
                                       const __nv_bfloat16* v, long long vs, const uint32_t* bits, int t, int lgC, float scale, float2 st,
                                       __nv_bfloat16* dq) {
  const int lane = threadIdx.x & 31;
  float acc[D / 32];
  bool gone = false;                                        // every column is NaN, whatever follows
#pragma unroll
  for (int y = 0; y < D / 32; ++y) acc[y] = 0.f;
  for (int leaf = 0; leaf <= (t >> lgC) && !gone; ++leaf) {
    if (!((bits[leaf >> 5] >> (leaf & 31)) & 1u)) continue;
    const int end = min((leaf + 1) << lgC, t + 1);
    for (int j0 = leaf << lgC; j0 < end && !gone; j0 += 32) {
      const int j = j0 + lane;
      float ds = 0.f;
      if (j < end) {
        float s = 0.f, dp = 0.f;
#pragma unroll 2
        for (int c = 0; c < D; c += 8) {
          float x[8], y[8];
          Elem<__nv_bfloat16>::load_chunk(q + c, x);
          Elem<__nv_bfloat16>::load_chunk(k + j * ks + c, y);
#pragma unroll
          for (int e = 0; e < 8; ++e) s = fmaf(x[e], y[e], s);
          Elem<__nv_bfloat16>::load_chunk(dout + c, x);
          Elem<__nv_bfloat16>::load_chunk(v + j * vs + c, y);
#pragma unroll
          for (int e = 0; e < 8; ++e) dp = fmaf(x[e], y[e], dp);
        }
        ds = ex2_approx(fmaf(s, scale * kLog2e, st.x)) * fmaf(dp, scale, st.y * scale);
        ds = __bfloat162float(__float2bfloat16_rn(ds));
      }
      for (int x = 0; x < min(32, end - j0); ++x) {
        const float dx = __shfl_sync(0xffffffffu, ds, x);
#pragma unroll
        for (int y = 0; y < D / 32; ++y) acc[y] = fmaf(dx, __bfloat162float(k[(long long)(j0 + x) * ks + lane + 32 * y]), acc[y]);
      }
      bool nan = true;
#pragma unroll
      for (int y = 0; y < D / 32; ++y) nan = nan && acc[y] != acc[y];
      gone = __all_sync(0xffffffffu, nan);
    }
  }
#pragma unroll
  for (int y = 0; y < D / 32; ++y) dq[lane + 32 * y] = __float2bfloat16_rn(acc[y]);
}

// Two tiles share every load of 64 keys and values.  TMEM, per tile: S at column 0, dP at 64, dQ at 128 (the second tile's
// at 256 and on).  The issuer walks the steps: for either tile the product its dS still owes, then the next S and dP.
// Floor per tile and 64 keys: 1 K cycles of the tensor pipe; measured 1.9 K.
template <int D, int C>
__global__ void __launch_bounds__(kBwdThreads2, 1)
qm_bwd_q_kernel(Geometry geo, Args a, const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_do,
                const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int KS = D / 64, SLAB = 128 * 128, TILE = KS * SLAB, HSLAB = 64 * 128, HALF = KS * HSLAB, NS = (D == 128) ? 3 : 6;
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* sQ = smem;                         // [2] (Q, dO)
  uint8_t* sKV = sQ + 4 * TILE;               // [NS] (K, V) of 64 keys
  __shared__ StepRing ring;
  __shared__ uint64_t q_full, q_empty, kv_full[NS], kv_empty[NS], s_full[2], p_full[2], o_full[2], o_empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail, s_again, s_items;          // s_again: a row came out not finite; s_items: this CTA's last item + 1

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  grid_dependency();
  if (a.gate.off_dense()) return;
  if (tid == 0) {
    ring_init(ring, 18);
    for (int i = 0; i < NS; ++i) { mbar_init(&kv_full[i], 1); mbar_init(&kv_empty[i], 1); }
    mbar_init(&q_full, 1); mbar_init(&q_empty, 1);
    for (int i = 0; i < 2; ++i) { mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 8); mbar_init(&o_full[i], 1); mbar_init(&o_empty[i], 8); }
    s_fail = s_again = s_items = 0;
    mbar_fence_init();
  }
  if (warp == 0) { tmem_alloc(&tmem_slot, 512); tmem_relinquish(); }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem = tmem_slot;
  const int G = geo.G, lgG = a.lgG, tpt = 128 >> lgG, lgC = a.lgC;
  bool dead = false;
  auto wait = [&](uint64_t* bar, uint32_t parity) {
    if (!dead && !mbar_try_wait(bar, parity) && !mbar_wait_bounded(bar, parity)) { dead = true; s_fail = 1; }
  };
  int n = 0;
  int4 e;

  if (warp == 3) {
    // ------------------------------------------------ scheduler
    for (bool ok = true; ok;) {
      int item = 0;
      if (lane == 0) item = atomicAdd(a.ctr + 1, 1);
      item = __shfl_sync(0xffffffffu, item, 0);
      if (item >= a.n_pairs) { ring_push(ring, n, make_int4(0, 0, kEnd, 0), &s_fail); break; }
      if (lane == 0) { a.chain[item] = s_items; s_items = item + 1; }
      const qmb::Loc loc = qmb::locate<qmb::kPairs>(geo, a, item);
      const int len = loc.q.len, W = (((len + C - 1) >> lgC) + 31) >> 5, tiles = (len + tpt - 1) / tpt, tile0 = loc.part * a.per;
      const uint32_t* tb = a.tbits + loc.q.up_off + ((long long)loc.h * W + lane) * tiles + tile0;
      const uint32_t w0 = lane < W ? tb[0] : 0u, w1 = (lane < W && a.per == 2 && tile0 + 1 < tiles) ? tb[1] : 0u;
      // last 64-key unit each tile needs (-1: none): the last leaf's last unit that starts no later than the tile's last token
      auto last_unit = [&](uint32_t w, int t_last) {
        const int leaf = __reduce_max_sync(0xffffffffu, w != 0u ? lane * 32 + 31 - __clz(w) : -1);
        return leaf < 0 ? -1 : min(leaf * (C / 64) + C / 64 - 1, t_last >> 6);
      };
      const int l0 = last_unit(w0, min(len, (tile0 + 1) * tpt) - 1), l1 = last_unit(w1, min(len, (tile0 + 2) * tpt) - 1);
      const int last = max(l0, l1);
      if (last < 0) { ok = ring_push(ring, n, make_int4(item, 0, kFirst | kLast | kEmpty, 0), &s_fail); continue; }
      int flags = kFirst;
      for (int w = 0; w < W && ok; ++w) {
        const uint32_t v0 = __shfl_sync(0xffffffffu, w0, w), v1 = __shfl_sync(0xffffffffu, w1, w);
        for (uint32_t m = v0 | v1; m != 0u && ok; m &= m - 1u) {
          const int bit = __ffs(m) - 1;
#pragma unroll
          for (int x = 0; x < C / 64; ++x) {
            const int u = (w * 32 + bit) * (C / 64) + x;
            const bool n0 = ((v0 >> bit) & 1u) && u <= l0, n1 = ((v1 >> bit) & 1u) && u <= l1;
            if (!(n0 || n1) || !ok) continue;
            flags |= (n0 ? kNeed0 : 0) | (n1 ? kNeed0 * 2 : 0) | (u == l0 && n0 ? kLast0 : 0) | (u == l1 && n1 ? kLast0 * 2 : 0) | (u == last ? kLast : 0);
            ok = ring_push(ring, n, make_int4(item, u, flags, 0), &s_fail);
            flags = 0;
          }
        }
      }
    }
  } else if (warp == 0) {
    // ------------------------------------------------ TMA producer
    int items = 0, step = 0;
    qmb::Loc loc;
    while (ring_pop(ring, n, e, &s_fail)) {
      if (e.z & kEmpty) continue;
      if (e.z & kFirst) {
        loc = qmb::locate<qmb::kPairs>(geo, a, e.x);
        if (items > 0) wait(&q_empty, (uint32_t)((items - 1) & 1));
        if (lane == 0 && !dead) {
          mbar_arrive_expect_tx(&q_full, (uint32_t)(2 * a.per * TILE));
          for (int x = 0; x < a.per; ++x)
            for (int ks = 0; ks < KS; ++ks) {
              const int t = loc.q.tok + (loc.part * a.per + x) * tpt;
              tma_load_4d(smem_u32(sQ + 2 * x * TILE + ks * SLAB), &tm_q, &q_full, ks * 64, loc.h * G, t, loc.q.batch);
              tma_load_4d(smem_u32(sQ + (2 * x + 1) * TILE + ks * SLAB), &tm_do, &q_full, ks * 64, loc.h * G, t, loc.q.batch);
            }
        }
        ++items;
      }
      const int s = step % NS;
      if (step >= NS) wait(&kv_empty[s], (uint32_t)((step / NS - 1) & 1));
      if (lane == 0 && !dead) {
        mbar_arrive_expect_tx(&kv_full[s], (uint32_t)(2 * HALF));
        for (int ks = 0; ks < KS; ++ks) {
          tma_load_4d(smem_u32(sKV + 2 * s * HALF + ks * HSLAB), &tm_k, &kv_full[s], ks * 64, loc.h, loc.q.tok + e.y * 64, loc.q.batch);
          tma_load_4d(smem_u32(sKV + (2 * s + 1) * HALF + ks * HSLAB), &tm_v, &kv_full[s], ks * 64, loc.h, loc.q.tok + e.y * 64, loc.q.batch);
        }
      }
      __syncwarp();
      ++step;
    }
  } else if (warp == 1) {
    // ------------------------------------------------ UMMA issuer
    const uint32_t idesc_s = make_idesc_bf16(128, 64, 0, 0), idesc_o = make_idesc_bf16(128, D, 0, 1);
    const uint32_t q_b = desc_lo(smem_u32(sQ), 0), k_s = desc_lo(smem_u32(sKV), 0), k_g = desc_lo(smem_u32(sKV), HSLAB);
    struct Owed { int stage; uint32_t parity; bool fresh, last; } owed[2];
    owed[0].stage = owed[1].stage = -1;
    uint32_t cnt[2] = {0u, 0u}, outs[2] = {0u, 0u};
    int step = 0, items = 0, prev = -1;                        // prev: stage of the previous step, not yet released
    int len = 0x7fffffff;
    bool fresh[2] = {true, true};
    auto product = [&](int x) {
      const Owed w = owed[x];
      wait(&p_full[x], w.parity);
      if (w.fresh) {
        if (outs[x] > 0u) wait(&o_empty[x], (outs[x] - 1u) & 1u);
        ++outs[x];
      }
      tcgen05_fence_after_sync();
      const uint32_t t = tmem + (uint32_t)(x * 256), b = k_g + (uint32_t)(2 * w.stage * (HALF >> 4));
      if (elect_one()) {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          umma_bf16_ts(t + 128u, t + (uint32_t)((kk >> 1) * 32 + (kk & 1) * 8), desc64(b + kk * (2048 >> 4)), idesc_o, (!w.fresh || kk > 0) ? 1u : 0u);
        if (w.last) umma_commit(&o_full[x]);
      }
      __syncwarp();
      owed[x].stage = -1;
    };
    auto release = [&](int stage) {
      if (elect_one()) umma_commit(&kv_empty[stage]);
      __syncwarp();
    };
    while (ring_pop(ring, n, e, &s_fail)) {
      if (e.z & kEmpty) {                                      // (the read-out of the item before must not wait for a later step)
#pragma unroll
        for (int x = 0; x < 2; ++x)
          if (owed[x].stage >= 0) product(x);
        if (prev >= 0) release(prev);
        prev = -1;
        continue;
      }
      const int s = step % NS;
      if (e.z & kFirst) {
        wait(&q_full, (uint32_t)(items & 1));
        if (a.seqs != nullptr) len = qmb::locate<qmb::kPairs>(geo, a, e.x).q.len;
        fresh[0] = fresh[1] = true;
        ++items;
      }
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (owed[x].stage >= 0) product(x);
        if (x == 1 && prev >= 0) release(prev);                // both tiles' products of the previous step are out
        if (!((e.z >> 4) & (1 << x))) continue;
        if (x == 0 || !(e.z & kNeed0)) {
          wait(&kv_full[s], (uint32_t)((step / NS) & 1));
          if (len - e.y * 64 < 64) {
            // packed: the keys past the sequence's end belong to its neighbour (their dS is zero, but a key that is not
            // finite would still reach the sum)
            zero_rows(sKV + 2 * s * HALF, HSLAB, KS, len - e.y * 64, 64);
            fence_proxy_async_smem();
            __syncwarp();
          }
        }
        tcgen05_fence_after_sync();
        const uint32_t q0 = q_b + (uint32_t)(2 * x * (TILE >> 4)), kv0 = k_s + (uint32_t)(2 * s * (HALF >> 4)), t = tmem + (uint32_t)(x * 256);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            umma_bf16(t, desc64(q0 + ((uint32_t)((kk >> 2) * SLAB + (kk & 3) * 32) >> 4)), desc64(kv0 + ((uint32_t)((kk >> 2) * HSLAB + (kk & 3) * 32) >> 4)),
                      idesc_s, kk > 0);
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            umma_bf16(t + 64u, desc64(q0 + (TILE >> 4) + ((uint32_t)((kk >> 2) * SLAB + (kk & 3) * 32) >> 4)),
                      desc64(kv0 + (HALF >> 4) + ((uint32_t)((kk >> 2) * HSLAB + (kk & 3) * 32) >> 4)), idesc_s, kk > 0);
          umma_commit(&s_full[x]);
        }
        __syncwarp();
        owed[x].stage = s; owed[x].parity = cnt[x]++ & 1u;
        owed[x].fresh = fresh[x]; owed[x].last = ((e.z >> 6) & (1 << x)) != 0;
        fresh[x] = false;
      }
      if ((e.z & kLast) && elect_one()) umma_commit(&q_empty);
      __syncwarp();
      prev = s;
      ++step;
    }
#pragma unroll
    for (int x = 0; x < 2; ++x)
      if (owed[x].stage >= 0) product(x);
  } else if (warp >= 4) {
    // ------------------------------------------------ dS and the read-out: a group of eight warps per tile
    const int x = (warp - 4) >> 3, part = ((warp - 4) >> 2) & 1, quarter = warp & 3;
    const int row = quarter * 32 + lane, head = row & (G - 1);
    const uint32_t lane_sel = (uint32_t)(quarter * 32) << 16;
    const uint32_t base = tmem + lane_sel + (uint32_t)(x * 256 + part * 32);
    const uint64_t sl2 = pack2(geo.scale * kLog2e, geo.scale * kLog2e), sc = pack2(geo.scale, geo.scale);
    int cnt = 0, outs = 0, t = 0, W = 0, wi = -1;
    bool live = false, any_step = false;
    float2 st = make_float2(-CUDART_INF_F, 0.f);
    uint32_t word = 0u, next = 0u;
    const uint32_t* bits = nullptr;
    qmb::Loc loc;
    while (ring_pop(ring, n, e, &s_fail)) {
      if (e.z & kFirst) {
        loc = qmb::locate<qmb::kPairs>(geo, a, e.x);
        t = (loc.part * a.per + x) * tpt + (row >> lgG);
        live = t < loc.q.len && x < a.per;
        W = (((loc.q.len + C - 1) >> lgC) + 31) >> 5;
        const long long r0 = (long long)loc.h * loc.q.len + (live ? t : 0);
        bits = a.bits + loc.q.bits_off + r0 * W;
        st = live ? a.stat[loc.q.leaf_off + r0 * G + head] : make_float2(-CUDART_INF_F, 0.f);
        wi = -1;
        any_step = false;
        next = live ? bits[0] : 0u;
      }
      if ((e.z >> 4) & (1 << x)) {
        const int leaf = (e.y * 64) >> lgC;
        if ((leaf >> 5) != wi) {
          const bool seq = (leaf >> 5) == wi + 1;
          wi = leaf >> 5;
          word = seq ? next : (live ? bits[wi] : 0u);
          next = (live && wi + 1 < W) ? bits[wi + 1] : 0u;     // in flight until the leaves of the next word come up
        }
        const bool sel = live && ((word >> (leaf & 31)) & 1u);
        const int nv = sel ? max(0, min(32, t - (e.y * 64 + part * 32) + 1)) : 0;   // visible keys of this warp's 32
        any_step = true;
        const int c = cnt++;
        wait(&s_full[x], (uint32_t)(c & 1));
        tcgen05_fence_after_sync();
        uint32_t dk[16];
        if (__any_sync(0xffffffffu, nv > 0)) {
          uint32_t rs[32], rp[32];
          tmem_ld_32x32(base, rs);
          tmem_ld_32x32(base + 64u, rp);
          const uint64_t bias = sel ? pack2(st.x, st.x) : pack2(-CUDART_INF_F, -CUDART_INF_F), nd = pack2(st.y * geo.scale, st.y * geo.scale);
          const bool fast = __all_sync(0xffffffffu, nv == 32 || !sel);
          tmem_ld_wait();
          auto run = [&](auto masked) {
#pragma unroll
            for (int y = 0; y < 16; ++y) {
              float p0, p1, d0, d1;
              prob_grad2(rs[2 * y], rs[2 * y + 1], rp[2 * y], rp[2 * y + 1], sl2, bias, sc, nd, p0, p1, d0, d1);
              if (masked.value) {
                if (2 * y >= nv) d0 = 0.f;
                if (2 * y + 1 >= nv) d1 = 0.f;
              }
              dk[y] = pack_bf16(d0, d1);
            }
          };
          if (fast) run(Bool<false>()); else run(Bool<true>());
        } else {
#pragma unroll
          for (int y = 0; y < 16; ++y) dk[y] = 0u;
        }
        tmem_st_32x16(base, dk);                               // over columns of S this warp has already read
        tmem_st_wait();
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[x]);
      }
      if (!(e.z & kLast)) continue;
      constexpr int CPW = D / 2;
      __nv_bfloat16* dst = a.dq + (long long)loc.q.batch * a.dq_s[0] + (long long)(loc.q.tok + t) * a.dq_s[1] +
                           (long long)(loc.h * G + head) * a.dq_s[2] + part * CPW;
      if (!any_step) {                                          // nothing selected by any row of the tile
        if (live)
#pragma unroll
          for (int y = 0; y < CPW; y += 8) *reinterpret_cast<uint4*>(dst + y) = make_uint4(0u, 0u, 0u, 0u);
        continue;
      }
      wait(&o_full[x], (uint32_t)(outs & 1));
      ++outs;
      tcgen05_fence_after_sync();
#pragma unroll
      for (int y = 0; y < CPW; y += 32) {
        uint32_t r[32];
        tmem_ld_32x32(tmem + lane_sel + (uint32_t)(x * 256 + 128 + part * CPW + y), r);
        tmem_ld_wait();
        if (y + 32 >= CPW) {
          tcgen05_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive(&o_empty[x]);
        }
        if (live) {
          if (!all_finite(r)) s_again = 1;
          store_row<32>(dst + y, r);
        }
      }
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(a.status, (int)PISA_ERR_TIMEOUT);
  if (warp == 0) tmem_dealloc(tmem, 512);
  if (!s_again || s_fail) return;
  for (int item = s_items - 1; item >= 0; item = a.chain[item] - 1) {
    const qmb::Loc loc = qmb::locate<qmb::kPairs>(geo, a, item);
    const int len = loc.q.len, W = (((len + C - 1) >> lgC) + 31) >> 5;
    const long long b = loc.q.batch, tok = loc.q.tok;
    for (int row = warp; row < 128 * a.per; row += kBwdThreads2 / 32) {
      const int t = loc.part * a.per * tpt + (row >> lgG), head = row & (G - 1), hq = loc.h * G + head;
      if (t >= len) break;
      __nv_bfloat16* dq = a.dq + b * a.dq_s[0] + (tok + t) * a.dq_s[1] + hq * a.dq_s[2];
      float finite = 0.f;
#pragma unroll
      for (int y = 0; y < D / 32; ++y) finite = fmaf(__bfloat162float(dq[lane + 32 * y]), 0.f, finite);
      if (!__any_sync(0xffffffffu, finite != finite)) continue;
      const long long r0 = (long long)loc.h * len + t;
      dq_row<D>(a.q + b * geo.qs[0] + (tok + t) * geo.qs[1] + hq * geo.qs[2], a.dout + b * geo.os[0] + (tok + t) * geo.os[1] + hq * geo.os[2],
                a.k + b * geo.ks[0] + tok * geo.ks[1] + loc.h * geo.ks[2], geo.ks[1], a.v + b * geo.vs[0] + tok * geo.vs[1] + loc.h * geo.vs[2],
                geo.vs[1], a.bits + loc.q.bits_off + r0 * W, t, lgC, geo.scale, a.stat[loc.q.leaf_off + r0 * G + head], dq);
    }
  }
}

// split sums -> bf16, dk and dv in one launch (blockIdx.y); n4: vectors of four
__global__ void __launch_bounds__(256) qm_bwd_convert_kernel(const float* dk_acc, const float* dv_acc, __nv_bfloat16* dk, __nv_bfloat16* dv,
                                                             long long n4, Gate gate) {
  grid_dependency();
  if (gate.off_dense()) return;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  const float4 x = reinterpret_cast<const float4*>(blockIdx.y ? dv_acc : dk_acc)[i];
  reinterpret_cast<uint2*>(blockIdx.y ? dv : dk)[i] = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
}
// ... and of the first blocks only: one block per (256 vectors of a block, KV head, sequence)
__global__ void __launch_bounds__(256) qm_bwd_convert0_kernel(Geometry geo, Args a) {
  grid_dependency();
  if (a.gate.off_dense()) return;
  const int i = blockIdx.x * 256 + threadIdx.x, d4 = geo.d / 4, key = i / d4, h = blockIdx.y;
  const qm::Seq q = a.seqs ? a.seqs[blockIdx.z] : qmb::seq_of(geo, a, blockIdx.z);
  if (key >= min(128, q.len)) return;
  const long long src = (((long long)q.pyr_row * geo.Hkv + h) * 128) * d4 + i, dst = ((q.cu + key) * geo.Hkv + h) * d4 + (i - key * d4);
  const float4 x = reinterpret_cast<const float4*>(a.dk_acc)[src], y = reinterpret_cast<const float4*>(a.dv_acc)[src];
  reinterpret_cast<uint2*>(a.dk)[dst] = make_uint2(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w));
  reinterpret_cast<uint2*>(a.dv)[dst] = make_uint2(pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
}

struct Maps { CUtensorMap q, dout, k, v, k64, v64; };

template <int D, int C>
int launch_dc(const Geometry& g, const Args& a, const Maps& m, long long tokens, cudaStream_t s) {
  const int W = ((g.N + C - 1) / C + 31) / 32, tpt = 128 / g.G;
  kernel_mark("bwd_prep", s);
  int st = launch_dependent<qm_bwd_prep_kernel<D>>("qm_bwd_prep", dim3((unsigned)a.n_tiles), 256u, (size_t)(tpt + 1) * W * 4, s, g, a);
  if (st != PISA_OK) return st;
  kernel_mark("bwd_kv", s);
  constexpr size_t tile = (size_t)(D / 64) * 128 * 128;
  st = launch_dependent<qm_bwd_kv_kernel<D, C>>("qm_bwd_kv", dim3((unsigned)(a.n_keys < num_sms() ? a.n_keys : num_sms())), kBwdThreads2,
                                                (2 + 2 * (D == 128 ? 2 : 4)) * tile + 1024, s, g, a, m.q, m.dout, m.k, m.v);
  if (st != PISA_OK) return st;
  kernel_mark("bwd_q", s);
  st = launch_dependent<qm_bwd_q_kernel<D, C>>("qm_bwd_q", dim3((unsigned)(a.n_pairs < num_sms() ? a.n_pairs : num_sms())), kBwdThreads2,
                                               (4 + (D == 128 ? 3 : 6)) * tile + 1024, s, g, a, m.q, m.dout, m.k64, m.v64);
  if (st != PISA_OK || (a.splits == 1 && a.splits0 == 1)) return st;
  kernel_mark("bwd_convert", s);
  if (a.splits == 1)
    return launch_dependent<qm_bwd_convert0_kernel>("qm_bwd_convert0", dim3((unsigned)(128 * D / 4 / 256), (unsigned)g.Hkv, (unsigned)(a.seqs ? a.nseq : g.B)),
                                                    256u, 0, s, g, a);
  const long long n4 = tokens * g.B * g.Hkv * g.d / 4;
  return launch_dependent<qm_bwd_convert_kernel>("qm_bwd_convert", dim3((unsigned)((n4 + 255) / 256), 2u), 256u, 0, s, (const float*)a.dk_acc,
                                                 (const float*)a.dv_acc, a.dk, a.dv, n4, a.gate);
}

}  // namespace

int launch_qm_bwd(const Geometry& g, const Args& a, const void* q, const void* k, const void* v, long long tokens, cudaStream_t s) {
  Maps m;
  const int tpt = 128 / g.G;
  if (!qm_map_rows(&m.q, q, g.d, g.Hq, tokens, g.B, g.qs, g.G, tpt) || !qm_map_rows(&m.dout, a.dout, g.d, g.Hq, tokens, g.B, g.os, g.G, tpt) ||
      !qm_map_rows(&m.k, k, g.d, g.Hkv, tokens, g.B, g.ks, 1, 128) || !qm_map_rows(&m.v, v, g.d, g.Hkv, tokens, g.B, g.vs, 1, 128) ||
      !qm_map_rows(&m.k64, k, g.d, g.Hkv, tokens, g.B, g.ks, 1, 64) || !qm_map_rows(&m.v64, v, g.d, g.Hkv, tokens, g.B, g.vs, 1, 64)) {
    record_cuda_error("qm_bwd tensor maps", cudaErrorInvalidValue);
    return PISA_ERR_CUDA;
  }
  if (g.d == 128) return g.C == 128 ? launch_dc<128, 128>(g, a, m, tokens, s) : launch_dc<128, 64>(g, a, m, tokens, s);
  return g.C == 128 ? launch_dc<64, 128>(g, a, m, tokens, s) : launch_dc<64, 64>(g, a, m, tokens, s);
}

}  // namespace pisa
