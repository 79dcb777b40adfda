// Packed variable-length batches through the query-major kernels (see query_major.cuh): no padding and no copies.  A table
// with one entry per sequence (its place in the packed tensors and in the score tables) is written to the workspace; every
// kernel maps its work items or rows to (sequence, position) through it.  One set of launches serves as many sequences as
// the workspace has room for score tables.
#include <algorithm>
#include <memory>
#include <new>

#include "launch.cuh"
#include "pisa_tensor.cuh"
#include "query_major.cuh"

namespace pisa {

namespace {

constexpr int kChunkSeqs = 256;
struct TableChunk {                       // a kernel parameter (18 KB): the table travels without a copy from host memory
  int n, first;
  qm::Seq seq[kChunkSeqs];
  qm::SeqOrder order[kChunkSeqs];
};

__global__ void __launch_bounds__(kChunkSeqs) qm_table_kernel(const __grid_constant__ TableChunk c, qm::Seq* seqs, qm::SeqOrder* order) {
  grid_dependency();
  const int i = threadIdx.x;
  if (i < c.n) {
    seqs[c.first + i] = c.seq[i];
    order[c.first + i] = c.order[i];
  }
}

// level 1 of every sequence's pyramid: one CTA per (leaf, KV head)
__global__ void __launch_bounds__(256) qm_packed_leaves_kernel(Geometry geo, const qm::Seq* seqs, int nseq, int lgC, int lgg,
                                                               const __nv_bfloat16* k, __nv_bfloat16* pyr) {
  __shared__ float red[16][128];
  grid_dependency();
  const int h = blockIdx.y, d = geo.d, chunks = d / 8;
  int lo_s = 0, hi_s = nseq;
  while (hi_s - lo_s > 1) {
    const int mid = (lo_s + hi_s) >> 1;
    if (seqs[mid].leaf0 <= (int)blockIdx.x) lo_s = mid; else hi_s = mid;
  }
  const qm::Seq q = seqs[lo_s];
  if (qm::top_level(q.len, lgC, lgg, geo.K) < 2) return;           // no level above the leaves is scored: no summaries kept
  const int leaf = (int)blockIdx.x - q.leaf0, M1 = (q.len + geo.C - 1) / geo.C;
  const int cx = threadIdx.x % chunks, ry = threadIdx.x / chunks, RY = min(16, (int)blockDim.x / chunks);
  const int lo = leaf * geo.C, hi = min(lo + geo.C, q.len);
  const __nv_bfloat16* base = k + (long long)q.tok * geo.ks[1] + (long long)h * geo.ks[2] + cx * 8;
  if (ry < RY) {
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    for (int r = lo + ry; r < hi; r += RY) {
      float x[8];
      Elem<__nv_bfloat16>::load_chunk(base + (long long)r * geo.ks[1], x);
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] += x[e];
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) red[ry][cx * 8 + e] = acc[e];
  }
  __syncthreads();
  for (int col = threadIdx.x; col < d; col += blockDim.x) {       // fixed-order reduction over the row groups
    float sum = 0.f;
    for (int r = 0; r < RY; ++r) sum += red[r][col];
    pyr[((long long)q.pyr_row + (long long)h * M1 + leaf) * d + col] = __float2bfloat16_rn(sum / (float)(hi - lo));
  }
}

// the levels above, from shared memory: one CTA per (16-byte column chunk, KV head, sequence)
__global__ void __launch_bounds__(128) qm_packed_levels_kernel(Geometry geo, const qm::Seq* seqs, int lgC, int lgg, __nv_bfloat16* pyr) {
  extern __shared__ uint4 s_rows[];
  grid_dependency();
  const qm::Seq q = seqs[blockIdx.z];
  const int cx = blockIdx.x, h = blockIdx.y, d = geo.d;
  const int top = qm::top_level(q.len, lgC, lgg, geo.K);           // scores need the levels below it
  if (top < 3) return;
  int Mb = qm::level_nodes(q.len, lgC, lgg, 1);
  uint4* src = s_rows;
  uint4* dst = s_rows + Mb;
  long long row0 = q.pyr_row;
  for (int i = threadIdx.x; i < Mb; i += blockDim.x)
    src[i] = *reinterpret_cast<const uint4*>(pyr + (row0 + (long long)h * Mb + i) * d + cx * 8);
  __syncthreads();
  for (int l = 2; l < top; ++l) {
    const int Ml = qm::level_nodes(q.len, lgC, lgg, l);
    row0 += (long long)geo.Hkv * Mb;
    for (int i = threadIdx.x; i < Ml; i += blockDim.x) {
      const int lo = i << lgg, hi = min(lo + (1 << lgg), Mb);
      float acc[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[e] = 0.f;
      for (int r = lo; r < hi; ++r) {
        float x[8];
        Elem<__nv_bfloat16>::load_chunk(reinterpret_cast<const __nv_bfloat16*>(src + r), x);
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] += x[e];
      }
      const float inv = 1.f / (float)(hi - lo);
      uint4 o;
      __nv_bfloat16* ov = reinterpret_cast<__nv_bfloat16*>(&o);
#pragma unroll
      for (int e = 0; e < 8; ++e) ov[e] = __float2bfloat16_rn(acc[e] * inv);
      dst[i] = o;
      *reinterpret_cast<uint4*>(pyr + (row0 + (long long)h * Ml + i) * d + cx * 8) = o;
    }
    __syncthreads();
    uint4* t = src; src = dst; dst = t;
    Mb = Ml;
  }
}

int log2i(int x) { return 31 - __builtin_clz((unsigned)x); }

// what one sequence adds to a launch
struct Need { size_t leaf, up, bits, pyr; int leaves, top; };
Need need_of(const Geometry& g, int len) {
  const int lgC = log2i(g.C), lgg = log2i(g.g);
  Need n;
  n.leaves = qm::level_nodes(len, lgC, lgg, 1);
  n.top = qm::top_level(len, lgC, lgg, g.K);
  const size_t rows = (size_t)len * g.Hkv;
  n.leaf = rows * qm::level_width(n.leaves) * g.G;
  n.up = rows * qm::table_width(len, lgC, lgg, n.top);
  n.bits = rows * ((n.leaves + 31) / 32);
  n.pyr = 0;
  for (int l = 1; l < n.top; ++l) n.pyr += (size_t)g.Hkv * qm::level_nodes(len, lgC, lgg, l);
  return n;
}
size_t bytes_of(const Geometry& g, const Need& n) {       // table entry and order included
  return n.leaf * 4 + n.up * 4 + n.bits * 4 + n.pyr * g.d * 2 + sizeof(qm::Seq) + sizeof(qm::SeqOrder);
}
constexpr size_t kFixedBytes = 4096;                       // alignment of the regions, the counter, one spare pyramid row

}  // namespace

int qm_write_table(const qm::Seq* seqs, const qm::SeqOrder* order, int n, qm::Seq* d_seqs, qm::SeqOrder* d_order, cudaStream_t s) {
  std::unique_ptr<TableChunk> chunk(new (std::nothrow) TableChunk);
  if (!chunk) return PISA_ERR_INVALID_ARG;
  for (int i0 = 0; i0 < n; i0 += kChunkSeqs) {
    chunk->first = i0;
    chunk->n = std::min(kChunkSeqs, n - i0);
    std::copy(seqs + i0, seqs + i0 + chunk->n, chunk->seq);
    std::copy(order + i0, order + i0 + chunk->n, chunk->order);
    const int st = launch_dependent<qm_table_kernel>("qm_table", dim3(1), kChunkSeqs, 0, s, *chunk, d_seqs, d_order);
    if (st != PISA_OK) return st;
  }
  return PISA_OK;
}

size_t qm_packed_bytes(const Geometry& g, int len) { return kFixedBytes + bytes_of(g, need_of(g, len)); }

// The sequences ids[0..n) (ascending) of a packed batch; g: the geometry of the call (heads, strides); every one of them
// fits the workspace alone (qm_packed_bytes).
int qm_forward_packed(const Geometry& g, const int32_t* cu, const int* ids, int n, long long total, const void* q, const void* k,
                      const void* v, int32_t* idx, void* out, float* lse, void* ws_, size_t ws_bytes, int32_t* status,
                      cudaStream_t s) {
  const int lgC = log2i(g.C), lgg = log2i(g.g);
  std::unique_ptr<TableChunk> chunk(new (std::nothrow) TableChunk);
  std::unique_ptr<int[]> by_len(new (std::nothrow) int[(size_t)n + 1]);
  std::unique_ptr<int[]> item0(new (std::nothrow) int[(size_t)n + 1]);
  if (!chunk || !by_len || !item0) return PISA_ERR_INVALID_ARG;
  for (int at = 0; at < n;) {
    size_t leaf = 0, up = 0, bits = 0, pyr = 0, used = kFixedBytes;
    long long rows = 0;
    int end = at, shortest = 0x7fffffff, leaves = 0, deepest = 0, most_leaves = 0;
    while (end < n) {                                      // as many sequences as the workspace takes
      const int len = cu[ids[end] + 1] - cu[ids[end]];
      const Need w = need_of(g, len);
      const size_t b = bytes_of(g, w);
      if (end > at && (used + b > ws_bytes || rows + len > (1LL << 24) || end - at >= 65535)) break;
      used += b; leaf += w.leaf; up += w.up; bits += w.bits; pyr += w.pyr;
      rows += len; leaves += w.leaves;
      shortest = std::min(shortest, len);
      deepest = std::max(deepest, w.top);
      most_leaves = std::max(most_leaves, w.leaves);
      ++end;
    }
    const int m = end - at;
    // regions
    char* p = (char*)ws_;
    auto take = [&](size_t bytes) { char* r = p; p += align_up(bytes, 256); return r; };
    qm::Args a = {};
    a.lgC = lgC; a.lgg = lgg; a.lgG = log2i(g.G);
    a.ctr = (int32_t*)take(256);
    qm::Seq* d_seqs = (qm::Seq*)take((size_t)m * sizeof(qm::Seq));
    qm::SeqOrder* d_order = (qm::SeqOrder*)take((size_t)m * sizeof(qm::SeqOrder));
    __nv_bfloat16* d_pyr = (__nv_bfloat16*)take((pyr + 1) * g.d * 2);
    a.leaf = (float*)take(leaf * 4);
    a.up = (float*)take(up * 4);
    a.bits = (uint32_t*)take(bits * 4);
    a.seqs = d_seqs; a.order = d_order; a.nseq = m;
    a.want_leaf = 1;
    a.status = status;
    a.tiles = qm_tiles_per_item(g, rows * g.Hkv);
    const int tpt = a.tiles * 128 / g.G;
    for (int i = 0; i < m; ++i) by_len[i] = i;
    std::stable_sort(by_len.get(), by_len.get() + m, [&](int x, int y) {
      return cu[ids[at + x] + 1] - cu[ids[at + x]] > cu[ids[at + y] + 1] - cu[ids[at + y]];
    });
    int items = 0;
    for (int i = 0; i < m; ++i) {
      const int len = cu[ids[at + by_len[i]] + 1] - cu[ids[at + by_len[i]]];
      item0[i] = items;
      items += g.Hkv * ((len + tpt - 1) / tpt);
    }
    a.n_items = items;
    // table
    kernel_mark("qm_table", s);
    long long o_leaf = 0, o_up = 0, o_bits = 0, o_pyr = 0, row0 = 0;
    int leaf0 = 0, st = PISA_OK;
    for (int i0 = 0; i0 < m; i0 += kChunkSeqs) {
      chunk->first = i0;
      chunk->n = std::min(kChunkSeqs, m - i0);
      for (int i = 0; i < chunk->n; ++i) {
        const int id = ids[at + i0 + i], len = cu[id + 1] - cu[id];
        const Need w = need_of(g, len);
        qm::Seq& e = chunk->seq[i];
        e.cu = cu[id]; e.leaf_off = o_leaf; e.up_off = o_up; e.bits_off = o_bits;
        e.tok = cu[id]; e.batch = 0; e.len = len; e.pyr_row = (int)o_pyr;
        e.row0 = (int)row0; e.leaf0 = leaf0;
        o_leaf += (long long)w.leaf; o_up += (long long)w.up; o_bits += (long long)w.bits; o_pyr += (long long)w.pyr;
        row0 += len;
        leaf0 += w.leaves;
        chunk->order[i].seq = by_len[i0 + i];
        chunk->order[i].item0 = item0[i0 + i];
      }
      st = launch_dependent<qm_table_kernel>("qm_table", dim3(1), kChunkSeqs, 0, s, *chunk, d_seqs, d_order);
      if (st != PISA_OK) return st;
    }
    // summaries of the levels that scores read (none when no sequence prunes above its leaves)
    if (deepest >= 2) {
      kernel_mark("qm_packed_pyramid", s);
      st = launch_dependent<qm_packed_leaves_kernel>("qm_packed_leaves", dim3((unsigned)leaves, (unsigned)g.Hkv), 256u, 0, s, g,
                                                     (const qm::Seq*)d_seqs, m, lgC, lgg, (const __nv_bfloat16*)k, d_pyr);
      if (st != PISA_OK) return st;
      if (deepest >= 3) {
        st = launch_dependent<qm_packed_levels_kernel>("qm_packed_levels", dim3((unsigned)(g.d / 8), (unsigned)g.Hkv, (unsigned)m), 128u,
                                                       (size_t)most_leaves * 2 * 16, s, g, (const qm::Seq*)d_seqs, lgC, lgg, d_pyr);
        if (st != PISA_OK) return st;
      }
    }
    kernel_mark("qm_score", s);
    if ((st = launch_qm_score(g, a, q, k, total, d_pyr, (long long)pyr + 1, s)) != PISA_OK) return st;
    kernel_mark("qm_select", s);
    if ((st = launch_qm_select_full(g, a, rows, idx, nullptr, lse, nullptr, s)) != PISA_OK) return st;
    kernel_mark("qm_attend", s);
    if ((st = launch_qm_attend(g, a, q, k, v, total, lse, out, shortest <= g.C, !tensor_path_supported(g, PISA_BF16), s)) != PISA_OK) return st;
    at = end;
  }
  return PISA_OK;
}

}  // namespace pisa
