// Host side of the dense masked backward (see qm_bwd.cuh).
#include <algorithm>
#include <memory>
#include <new>

#include "launch.cuh"
#include "pisa_tensor.cuh"
#include "qm_bwd.cuh"

namespace pisa {

namespace {

int log2i(int x) { return 31 - __builtin_clz((unsigned)x); }

// tokens of all sequences, leaf-bit words, 128-row tiles' words and tiles summed over them (per KV head)
struct Sizes { size_t rows, words, twords, tiles; };
struct Layout { size_t ctr, chain, bits, tbits, stat, acc, total; };
// acc: room for the split sums, of all keys (kAccAll) or of the first blocks of `acc` sequences
enum { kAccAll = -1 };
Layout layout(const Geometry& g, const Sizes& z, long long acc) {
  Layout l;
  size_t o = 0;
  l.ctr = o; o += 256;
  l.chain = o; o += align_up(z.tiles * g.Hkv * 4, 256);
  l.bits = o; o += align_up(z.words * g.Hkv * 4, 256);
  l.tbits = o; o += align_up(z.twords * g.Hkv * 4, 256);
  l.stat = o; o += align_up(z.rows * g.Hq * 8, 256);
  l.acc = o;
  const size_t acc_rows = acc == kAccAll ? z.rows : (size_t)acc * 128;
  o += 2 * align_up(acc_rows * g.Hkv * g.d * 4, 256);
  l.total = o;
  return l;
}
Sizes seq_sizes(const Geometry& g, int len) {
  const int tpt = 128 / g.G;
  const size_t W = ((len + g.C - 1) / g.C + 31) / 32, tiles = (size_t)((len + tpt - 1) / tpt);
  return {(size_t)len, (size_t)len * W, tiles * W, tiles};
}
Sizes uniform_sizes(const Geometry& g) {
  const Sizes z = seq_sizes(g, g.N);
  return {g.B * z.rows, g.B * z.words, g.B * z.twords, g.B * z.tiles};
}
// splits, splits0 and the room for their sums
struct Split { int all, first; long long acc; };
Split uniform_split(const Geometry& g) {
  Split x;
  x.all = qm_bwd_splits((long long)g.B * g.Hkv * ((g.N + 127) / 128));
  x.first = qm_bwd_splits0(((long long)g.N * g.G + 127) / 128, x.all);
  x.acc = x.all > 1 ? (long long)kAccAll : x.first > 1 ? g.B : 0;
  return x;
}
size_t table_bytes(size_t n) { return align_up(n * sizeof(qm::Seq), 256) + align_up(n * sizeof(qm::SeqOrder), 256); }

// Steps (128-row tile x 128 keys) per tile and selected block up to which the dense kernels win, in eighths: a dense step takes
// 7.2 K (d = 64) to 8.1 K SM cycles, 128 rows of the lists 7 to 7.5 K and 0.15 ms of preparation, inversion and conversions at
// 6000 tokens.  Whole calls in us, dense / lists (steps per tile and block in parentheses): 16 heads, G = 4, C = 64, K = 16: 3000
// tokens 213 / 291, 6000 483 / 471 (1.1), 12288 1097 / 879 (1.35); 32 heads, fan-in 4: 6000 891 / 836; C = 128, K = 32, 32 heads:
// 6000 1135 / 1143 (0.7), 12288 3961 / 2617 (1.25); 16 heads without groups: 6000 570 / 801, 12288 1749 / 1485 (2.2); 16 heads
// per group, d = 64, K = 8: 16384 919 / 1172, 32768 1943 / 2233 (1.0).
int steps_per_block8(const Geometry& g) {
  if (g.G == 1) return g.C == 128 ? 9 : 13;
  if (g.G == 16) return g.C == 128 ? 8 : 10;
  return g.C == 128 ? 6 : 8;
}

}  // namespace

// Parts that the rows of one 128-key block are dealt out to: a short sequence has few key blocks, and without parts a few
// SMs would work through all rows.
int qm_bwd_splits(long long key_items) {
  const long long want = 3LL * num_sms();
  return (int)std::max(1LL, std::min(8LL, (want + key_items - 1) / std::max(1LL, key_items)));
}
// ... and of the first block: about 96 tiles per part
int qm_bwd_splits0(long long tiles_of_longest, int splits) {
  return (int)std::max<long long>(splits, std::min(64LL, (tiles_of_longest + 95) / 96));
}
// Two tiles per item of the q kernel share their keys and values; one where pairs would leave SMs idle.
int qm_bwd_tiles_per_item(long long tiles) { return tiles >= 2LL * num_sms() ? 2 : 1; }

bool qm_bwd_supported(const Geometry& g, int dtype) {
  return dtype == PISA_BF16 && (g.d == 64 || g.d == 128) && (g.C == 64 || g.C == 128) && g.M[1] <= 1024 &&
         tma_strides(g.qs) && tma_strides(g.os);                    // (keys and values are read through tensor maps on either path)
}
// (a tile has N / 256 steps on average when it needs all key blocks)
int qm_bwd_always(const Geometry& g) { return 32 * g.K * steps_per_block8(g); }
// In a packed batch the dense kernels take all sequences at once and the lists one after the other: twelve sequences of 16 to
// 6000 tokens, 32 heads, fan-in 4 take 1.20 ms with all of them dense, 1.33 with those above 4096 tokens on the lists.
int qm_bwd_packed_longest(const Geometry& g) { return 32 * g.K * (g.G == 1 ? (g.C == 128 ? 19 : 24) : (g.C == 128 ? 12 : 15)); }

size_t qm_bwd_workspace_bytes(const Geometry& g) { return layout(g, uniform_sizes(g), uniform_split(g).acc).total; }

int qm_bwd(const Geometry& g, const void* q, const void* k, const void* v, const int32_t* idx, const void* out, const float* lse,
           const void* dout, void* dq, void* dk, void* dv, void* ws_, int32_t* status, Gate* gate, const float2** stat,
           cudaStream_t s) {
  char* ws = (char*)ws_;
  const int tpt = 128 / g.G, units = g.B * g.Hkv;
  qmb::Args a = {};
  const Split split = uniform_split(g);
  a.splits = split.all;
  a.splits0 = split.first;
  const Layout l = layout(g, uniform_sizes(g), split.acc);
  a.lgC = log2i(g.C); a.lgG = log2i(g.G);
  a.n_tiles = units * ((g.N + tpt - 1) / tpt);
  a.per = qm_bwd_tiles_per_item(a.n_tiles);
  a.n_pairs = units * ((g.N + a.per * tpt - 1) / (a.per * tpt));
  a.n_keys = units * (a.splits0 + ((g.N + 127) / 128 - 1) * a.splits);
  a.bits = (uint32_t*)(ws + l.bits); a.tbits = (uint32_t*)(ws + l.tbits); a.stat = (float2*)(ws + l.stat);
  a.chain = (int32_t*)(ws + l.chain); a.q = (const __nv_bfloat16*)q; a.k = (const __nv_bfloat16*)k; a.v = (const __nv_bfloat16*)v;
  a.idx = idx; a.lse = lse; a.out = (const __nv_bfloat16*)out; a.dout = (const __nv_bfloat16*)dout;
  a.dq = (__nv_bfloat16*)dq; a.dk = (__nv_bfloat16*)dk; a.dv = (__nv_bfloat16*)dv;
  a.dq_s[0] = (long long)g.N * g.Hq * g.d; a.dq_s[1] = (long long)g.Hq * g.d; a.dq_s[2] = g.d;
  a.ctr = (int32_t*)(ws + l.ctr); a.status = status;
  if (gate != nullptr) {
    *stat = a.stat;
    a.count = (uint32_t*)a.ctr + 4;
    const long long limit = (long long)a.n_tiles * g.K * steps_per_block8(g) / 8;
    *gate = Gate{a.count, (uint32_t)std::min<long long>(limit, 0xfffffffeLL)};
    a.gate = *gate;
    const cudaError_t e = cudaMemsetAsync(a.count, 0, 4, s);
    if (e != cudaSuccess) { record_cuda_error("step count memset", e); return PISA_ERR_CUDA; }
  }
  if (l.total > l.acc) {
    a.dk_acc = (float*)(ws + l.acc);
    a.dv_acc = a.dk_acc + (l.total - l.acc) / 8;
    const cudaError_t e = cudaMemsetAsync(a.dk_acc, 0, l.total - l.acc, s);
    if (e != cudaSuccess) { record_cuda_error("gradient memset", e); return PISA_ERR_CUDA; }
  }
  return launch_qm_bwd(g, a, q, k, v, g.N, s);
}

// ---------------------------------------------------------------- packed batches

size_t qm_bwd_packed_bytes(const Geometry& g, int len) { return table_bytes(1) + layout(g, seq_sizes(g, len), 1).total; }

int qm_bwd_packed(const Geometry& g, const int32_t* cu, const int* ids, int n, long long total, const void* q, const void* k,
                  const void* v, const int32_t* idx, const void* out, const float* lse, const void* dout, void* dq, void* dk,
                  void* dv, void* ws_, size_t ws_bytes, int32_t* status, cudaStream_t s) {
  std::unique_ptr<qm::Seq[]> seqs(new (std::nothrow) qm::Seq[(size_t)n]);
  std::unique_ptr<qm::SeqOrder[]> order(new (std::nothrow) qm::SeqOrder[(size_t)n]);
  std::unique_ptr<int[]> by_len(new (std::nothrow) int[(size_t)n]);
  if (!seqs || !order || !by_len) return PISA_ERR_INVALID_ARG;
  const int tpt = 128 / g.G;
  for (int at = 0; at < n;) {
    Sizes z = {0, 0, 0, 0};
    int end = at, longest = 0;
    long long tiles = 0, key_items = 0;
    while (end < n) {                                       // as many sequences as the workspace takes
      const int len = cu[ids[end] + 1] - cu[ids[end]];
      const Sizes w = seq_sizes(g, len), sum = {z.rows + w.rows, z.words + w.words, z.twords + w.twords, z.tiles + w.tiles};
      if (end > at && (table_bytes((size_t)(end - at + 1)) + layout(g, sum, end - at + 1).total > ws_bytes ||
                       sum.rows * g.Hq > (1ull << 30) || end - at >= 65535)) break;
      z = sum;
      tiles += (long long)g.Hkv * ((len + tpt - 1) / tpt);
      key_items += (long long)g.Hkv * ((len + 127) / 128);
      longest = std::max(longest, len);
      ++end;
    }
    const int m = end - at;
    qmb::Args a = {};
    // (the split sums of all keys are indexed like the pack, so only where its sequences run in one go and there is room)
    const size_t base = table_bytes((size_t)m) + layout(g, z, 0).total;
    const size_t all = 2 * align_up((size_t)total * g.Hkv * g.d * 4, 256);
    a.splits = (at == 0 && end == n && base + all <= ws_bytes) ? qm_bwd_splits(key_items) : 1;
    a.splits0 = qm_bwd_splits0((longest + tpt - 1) / tpt, a.splits);
    const size_t acc = a.splits > 1 ? all : a.splits0 > 1 ? 2 * align_up((size_t)m * 128 * g.Hkv * g.d * 4, 256) : 0;
    a.per = qm_bwd_tiles_per_item(tiles);
    char* ws = (char*)ws_;
    qm::Seq* d_seqs = (qm::Seq*)ws;
    qm::SeqOrder* d_order = (qm::SeqOrder*)(ws + align_up((size_t)m * sizeof(qm::Seq), 256));
    ws += table_bytes((size_t)m);
    const Layout l = layout(g, z, 0);
    long long words = 0, twords = 0, rows = 0;
    for (int i = 0; i < m; ++i) {
      const int id = ids[at + i], len = cu[id + 1] - cu[id];
      const Sizes w = seq_sizes(g, len);
      qm::Seq& e = seqs[i];
      e.cu = cu[id]; e.tok = cu[id]; e.batch = 0; e.len = len;
      e.bits_off = words; e.up_off = twords; e.leaf_off = rows * g.Hq;
      e.pyr_row = i; e.row0 = (int)rows; e.leaf0 = 0;
      words += (long long)w.words * g.Hkv; twords += (long long)w.twords * g.Hkv; rows += len;
      by_len[i] = i;
    }
    std::stable_sort(by_len.get(), by_len.get() + m, [&](int x, int y) { return seqs[x].len > seqs[y].len; });
    int i0 = 0, it = 0, ik = 0;
    for (int i = 0; i < m; ++i) {
      const int len = seqs[by_len[i]].len;
      order[i] = qm::SeqOrder{by_len[i], i0, it, ik};
      i0 += g.Hkv * ((len + a.per * tpt - 1) / (a.per * tpt));
      it += g.Hkv * ((len + tpt - 1) / tpt);
      ik += g.Hkv * (a.splits0 + ((len + 127) / 128 - 1) * a.splits);
    }
    kernel_mark("qm_table", s);
    int st = qm_write_table(seqs.get(), order.get(), m, d_seqs, d_order, s);
    if (st != PISA_OK) return st;
    a.seqs = d_seqs; a.order = d_order; a.nseq = m;
    a.lgC = log2i(g.C); a.lgG = log2i(g.G);
    a.n_pairs = i0; a.n_tiles = it; a.n_keys = ik;
    a.bits = (uint32_t*)(ws + l.bits); a.tbits = (uint32_t*)(ws + l.tbits); a.stat = (float2*)(ws + l.stat);
    a.chain = (int32_t*)(ws + l.chain); a.q = (const __nv_bfloat16*)q; a.k = (const __nv_bfloat16*)k; a.v = (const __nv_bfloat16*)v;
    a.idx = idx; a.lse = lse; a.out = (const __nv_bfloat16*)out; a.dout = (const __nv_bfloat16*)dout;
    a.dq = (__nv_bfloat16*)dq; a.dk = (__nv_bfloat16*)dk; a.dv = (__nv_bfloat16*)dv;
    a.dq_s[0] = 0; a.dq_s[1] = (long long)g.Hq * g.d; a.dq_s[2] = g.d;
    a.ctr = (int32_t*)(ws + l.ctr); a.status = status;
    if (acc > 0) {
      a.dk_acc = (float*)(ws + l.total);
      a.dv_acc = a.dk_acc + acc / 8;
      const cudaError_t e = cudaMemsetAsync(a.dk_acc, 0, acc, s);
      if (e != cudaSuccess) { record_cuda_error("gradient memset", e); return PISA_ERR_CUDA; }
    }
    Geometry gl = g;                                        // (the preparation sizes its shared memory by the longest sequence)
    gl.N = longest;
    if ((st = launch_qm_bwd(gl, a, q, k, v, total, s)) != PISA_OK) return st;
    at = end;
  }
  return PISA_OK;
}

}  // namespace pisa
