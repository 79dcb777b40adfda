// Which blocks a query tile's rows share (shared.cuh).  One CTA per tile: a counter per block in shared memory, the blocks that
// enough tokens selected in ascending order, and who selected them.  Bound by the two passes over the rows (L2): 0.3 ms for 33
// million entries.
#include "pisa_tensor.cuh"
#include "shared.cuh"
#include "tma_map.cuh"

namespace pisa {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxBlocks = 32768;              // counters of a tile: a byte per block in shared memory

// SLOTS: the place of the block in each token's row (bytes), else a mask of the tokens
template <bool SLOTS>
__global__ void __launch_bounds__(kThreads) shared_plan_kernel(Geometry geo, const int32_t* __restrict__ idx, SharedPlan p, int always0) {
  extern __shared__ uint32_t s_cnt[];                        // a byte per block: how many tokens selected it, then its place + 1
  __shared__ uint32_t s_who[SLOTS ? 1 : kSharedMax * 4];
  __shared__ uint32_t s_taken[128];
  __shared__ int s_n, s_warp[kThreads / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tpt = 128 / geo.G, tile = blockIdx.x, bh = blockIdx.y, K = geo.K, span = p.span;
  const int t0 = tile * tpt, nt = min(tpt, geo.N - t0);
  const int blocks = (t0 + nt - 1) / span + 1;               // visible to the tile's last token
  uint8_t* cnt8 = reinterpret_cast<uint8_t*>(s_cnt);
  for (int i = tid; i < (blocks + 3) / 4; i += kThreads) s_cnt[i] = 0u;
  if (!SLOTS)
    for (int i = tid; i < kSharedMax * 4; i += kThreads) s_who[i] = 0u;
  if (tid < 128) s_taken[tid] = 0u;
  if (tid == 0) s_n = 0;
  __syncthreads();
  const int32_t* rows = idx + ((long long)bh * geo.N + t0) * K;
  for (int e = tid; e < nt * K; e += kThreads) {
    const int node = rows[e];
    if (node >= 0 && node <= (t0 + e / K) / span) atomicAdd(&s_cnt[node >> 2], 1u << (8 * (node & 3)));
  }
  __syncthreads();
  const long long slot0 = ((long long)bh * p.tiles + tile) * p.max_nodes;
  for (int l0 = 0; l0 < blocks; l0 += kThreads) {
    const int node = l0 + tid;
    const bool hot = node < blocks && (cnt8[node] >= p.threshold || (always0 && node == 0 && cnt8[0] > 0));
    const unsigned bal = __ballot_sync(0xffffffffu, hot);
    if (lane == 0) s_warp[warp] = __popc(bal);
    __syncthreads();
    int place = s_n;
    for (int w = 0; w < warp; ++w) place += s_warp[w];
    place += __popc(bal & ((1u << lane) - 1u));
    const bool fits = hot && place < p.max_nodes;
    if (node < blocks) cnt8[node] = fits ? (uint8_t)(place + 1) : (uint8_t)0;
    if (fits) p.node[slot0 + place] = (uint16_t)node;
    __syncthreads();
    if (tid == 0)
      for (int w = 0; w < kThreads / 32; ++w) s_n += s_warp[w];
    __syncthreads();
  }
  const int n = min(s_n, p.max_nodes);
  uint8_t* slots = SLOTS ? p.slot + slot0 * tpt : nullptr;
  if (SLOTS) {
    for (int i = tid; i < n * tpt; i += kThreads) slots[i] = 255;
    __syncthreads();                                         // (the CTA's own stores: ordered by the barrier)
  }
  for (int e = tid; e < nt * K; e += kThreads) {
    const int node = rows[e], tl = e / K;
    if (node < 0 || node > (t0 + tl) / span) continue;
    const int place = (int)cnt8[node] - 1;
    if (place < 0) continue;
    if (SLOTS) slots[place * tpt + tl] = (uint8_t)(e - tl * K);
    else atomicOr(&s_who[place * p.words + (tl >> 5)], 1u << (tl & 31));
    atomicOr(&s_taken[tl], 1u << (e - tl * K));
  }
  __syncthreads();
  if (!SLOTS)
    for (int i = tid; i < n * p.words; i += kThreads) p.mask[slot0 * p.words + i] = s_who[i];
  if (tid < nt) p.taken[(long long)bh * geo.N + t0 + tid] = s_taken[tid];
  if (tid == 0) p.count[(long long)bh * p.tiles + tile] = n;
}

}  // namespace

bool shared_supported(const Geometry& g, int dtype, int blocks) {
  if (dtype != PISA_BF16 || (g.d != 128 && g.d != 64) || (g.C != 64 && g.C != 128)) return false;
  if (g.G > 16 || (g.G & (g.G - 1)) != 0 || g.K > kMaxK || blocks > kMaxBlocks) return false;
  for (int i = 0; i < 3; ++i)
    if ((g.qs[i] * 2) % 16 || (g.ks[i] * 2) % 16 || (g.vs[i] * 2) % 16) return false;
  if (!tma_strides(g.qs) || !tma_strides(g.ks) || !tma_strides(g.vs)) return false;
  const int tpt = 128 / g.G;
  if ((long long)g.B * g.Hkv > 65535 || (long long)g.B * g.Hkv * ((g.N + tpt - 1) / tpt) > 0x7fffffffLL) return false;
  return tma::encoder() != nullptr;
}

int launch_shared_plan(const Geometry& g, const int32_t* rows, const SharedPlan& plan, bool always0, cudaStream_t s) {
  const dim3 grid((unsigned)plan.tiles, (unsigned)(g.B * g.Hkv));
  const size_t smem = (size_t)((g.N + plan.span - 1) / plan.span + 3) / 4 * 4;
  if (plan.slot != nullptr) shared_plan_kernel<true><<<grid, kThreads, smem, s>>>(g, rows, plan, always0 ? 1 : 0);
  else shared_plan_kernel<false><<<grid, kThreads, smem, s>>>(g, rows, plan, always0 ? 1 : 0);
  return check_launch("shared_plan");
}

}  // namespace pisa
