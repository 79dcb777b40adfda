// Host side of the query-major kernels (see query_major.cuh): what they support, when they are the better choice, their
// workspace, and the sequence of launches.
#include "pisa_tensor.cuh"
#include "query_major.cuh"

namespace pisa {

namespace {

constexpr int kDenseMaxTokens = 32768;                 // 256 steps of 128 keys: the attention kernel's step lists
constexpr size_t kDenseMaxBytes = (size_t)4 << 30;     // score tables (they grow with N * M1)

constexpr int kStage1MaxG = 4;
// node table of one range of tokens (list-driven path): the larger the better -- at the headline shape 48 MB, inside L2,
// 7.5 ms for the stage, 256 MB 5.1, 1 GB 4.1 (each range is two launches that fill and drain the GPU)
constexpr size_t kSlabBytes = (size_t)1 << 30;

int log2i(int x) { return 31 - __builtin_clz((unsigned)x); }

struct Layout { size_t ctr, leaf, up, bits, total; };
Layout layout(const Geometry& g) {
  const int lgC = log2i(g.C), lgg = log2i(g.g);
  const int top = qm::top_level(g.N, lgC, lgg, g.K);
  const size_t rows = (size_t)g.B * g.Hkv * g.N;
  Layout l;
  size_t o = 0;
  l.ctr = o; o += 256;
  l.leaf = o; o += align_up(rows * qm::level_width(g.M[1]) * g.G * 4, 256);
  l.up = o; o += align_up(rows * qm::table_width(g.N, lgC, lgg, top) * 4, 256);
  l.bits = o; o += align_up(rows * ((g.M[1] + 31) / 32) * 4, 256);
  l.total = o;
  return l;
}

qm::Args uniform_args(const Geometry& g, char* ws, const Layout& l, int32_t* status) {
  qm::Args a = {};
  a.lgC = log2i(g.C); a.lgg = log2i(g.g); a.lgG = log2i(g.G);
  a.t0 = 0; a.t1 = g.N;
  a.tiles = qm_tiles_per_item(g, (long long)g.B * g.Hkv * g.N);
  const int tpt = a.tiles * 128 / g.G;
  a.n_items = g.B * g.Hkv * ((g.N + tpt - 1) / tpt);
  a.want_leaf = 1;
  a.leaf = (float*)(ws + l.leaf); a.up = (float*)(ws + l.up); a.bits = (uint32_t*)(ws + l.bits);
  a.ctr = (int32_t*)(ws + l.ctr);
  a.status = status;
  return a;
}

}  // namespace

// Two tiles per work item halve the key / value traffic, which bounds the dense kernels, once there are enough pairs for
// three waves of one item per SM (16 heads: 4096 tokens 206 us with one tile per item, 270 with two; 8192: 606 and 576).
int qm_tiles_per_item(const Geometry& g, long long unit_tokens) {
  return unit_tokens * g.G / 256 >= 3LL * num_sms() ? 2 : 1;
}

// Strides a tensor map can hold: below 2^40 bytes, not negative (the other kernels that read queries gather rows by pointer
// and take any).
bool tma_strides(const long long* st) {
  for (int i = 0; i < 3; ++i)
    if (st[i] < 0 || st[i] >= (1LL << 39)) return false;
  return true;
}

bool qm_supported(const Geometry& g, int dtype) {
  if (dtype != PISA_BF16 || g.score_mode != PISA_SCORE_LSE) return false;
  if (!tma_strides(g.qs) || !tma_strides(g.ks) || !tma_strides(g.vs)) return false;
  if ((g.d != 64 && g.d != 128) || (g.C != 64 && g.C != 128)) return false;
  return g.g == 2 || g.g == 4;
}

// Where the dense kernels win.  They cost a row N / 2 keys whatever it selects; the lists cost it K (token, block) pairs, so
// the line lies at a length proportional to K.  Whole forwards in us, dense / lists, of passages on 32 topics (neighbours
// select much the same leaves, which the lists' attention serves query-major: with queries that share nothing the lists take
// a third longer and the lines lie 1.5 times higher): G = 4, C = 64, K = 16: 12288 tokens 745 / 748 (16 heads), 1402 / 1265
// (32 heads, fan-in 4), 8192 763 / 838; G = 4, C = 128, K = 32: 12288 1744 / 2100, 16384 2964 / 2869; 16 KV heads without
// groups, K = 16: 16384 1612 / 1740, 24000 3304 / 2846; G = 16, d = 64, K = 8: 6000 331 / 367, 8192 526 / 461.  Shapes that
// the lists do not take stay dense further: their alternative is the exact fp32 path.  So do small problems, which the lists'
// eighteen launches weigh on (host tensors, 16384 tokens, one KV head of four query heads at a time: 3.13 ms dense, 3.21 lists).
bool qm_dense_preferred(const Geometry& g, int dtype) {
  if (!qm_supported(g, dtype) || g.M[1] > 512 || g.N > kDenseMaxTokens) return false;
  int per_block = g.G == 1 ? 1120 : g.C == 128 ? 480 : g.G == 16 ? 832 : 704;
  if (!tensor_path_supported(g, dtype) || (long long)g.B * g.Hq * g.N < (1 << 17)) per_block = g.G == 1 ? 2048 : g.C == 128 ? 704 : 1024;
  return g.N <= g.K * per_block && layout(g).total <= kDenseMaxBytes;
}

size_t qm_workspace_bytes(const Geometry& g) { return layout(g).total; }

// pyramid -> idx (and, where given, margins, row denominators, per-leaf denominators)
int qm_route(const Geometry& g, const void* q, const void* k, const void* pyramid, int32_t* idx, float* sel_lse,
             float* margin, float* lse_out, void* ws_, int32_t* status, cudaStream_t s) {
  char* ws = (char*)ws_;
  const Layout l = layout(g);
  const qm::Args a = uniform_args(g, ws, l, status);
  kernel_mark("qm_score", s);
  const long long pyr_rows = g.level_off[g.L] / g.d + (long long)g.B * g.Hkv * g.M[g.L];
  int st = launch_qm_score(g, a, q, k, g.N, pyramid, pyr_rows, s);
  if (st != PISA_OK) return st;
  kernel_mark("qm_select", s);
  return launch_qm_select_full(g, a, (long long)g.B * g.N, idx, margin, lse_out, sel_lse, s);
}

// attention over what qm_route just selected (its bits are in the workspace); lse: the rows' denominators
int qm_attend(const Geometry& g, const void* q, const void* k, const void* v, void* out, const float* lse, void* ws_,
              int32_t* status, cudaStream_t s) {
  char* ws = (char*)ws_;
  const Layout l = layout(g);
  const qm::Args a = uniform_args(g, ws, l, status);
  kernel_mark("qm_attend", s);
  // (where the lists do not take the problem its alternative is the exact fp32 path)
  return launch_qm_attend(g, a, q, k, v, g.N, lse, out, g.N <= g.C, !tensor_path_supported(g, PISA_BF16), s);
}

// ---------------------------------------------------------------- upper levels and final selection of the list-driven path

static long long stage1_slab(const Geometry& g, size_t scratch_bytes, int width) {
  const size_t per_token = (size_t)g.B * g.Hkv * width * 4;
  const size_t bytes = scratch_bytes < kSlabBytes ? scratch_bytes : kSlabBytes;
  return (long long)(bytes / per_token) / 256 * 256;         // whole work items of two tiles
}

bool qm_stage1_preferred(const Geometry& g, int dtype, size_t scratch_bytes) {
  // (groups of more than four heads: the per-token scoring shares its gathered summaries among them, 0.68 ms against 1.3
  // at 65536 tokens, 2 KV heads of 16 query heads; beyond 2048 leaves it costs log N per token and this N)
  if (!qm_supported(g, dtype) || g.L < 2 || g.M[1] > 2048 || g.G > kStage1MaxG) return false;
  const int lgC = log2i(g.C), lgg = log2i(g.g), top = qm::top_level(g.N, lgC, lgg, g.K);
  const int width = qm::table_width(g.N, lgC, lgg, top);
  return width == 0 || stage1_slab(g, scratch_bytes, width) > 0;
}

int qm_stage1(const Geometry& g, const void* q, const void* pyramid, int32_t* par, float* margin, float* scratch,
              size_t scratch_bytes, int32_t* status, cudaStream_t s) {
  qm::Args a = {};
  a.lgC = log2i(g.C); a.lgg = log2i(g.g); a.lgG = log2i(g.G);
  a.up = scratch; a.status = status;
  const int width = qm::table_width(g.N, a.lgC, a.lgg, qm::top_level(g.N, a.lgC, a.lgg, g.K));
  const long long slab = width == 0 ? g.N : stage1_slab(g, scratch_bytes, width);
  const long long pyr_rows = g.level_off[g.L] / g.d + (long long)g.B * g.Hkv * g.M[g.L];
  for (long long t0 = 0; t0 < g.N; t0 += slab) {
    a.t0 = (int)t0;
    a.t1 = (int)(t0 + slab < g.N ? t0 + slab : g.N);
    a.tiles = qm_tiles_per_item(g, (long long)g.B * g.Hkv * (a.t1 - a.t0));
    const int tpt = a.tiles * 128 / g.G;
    a.n_items = g.B * g.Hkv * ((a.t1 - a.t0 + tpt - 1) / tpt);
    int st = PISA_OK;
    if (width > 0) st = launch_qm_score(g, a, q, nullptr, g.N, pyramid, pyr_rows, s);
    if (st == PISA_OK) st = launch_qm_select_stage1(g, a, (long long)g.B * (a.t1 - a.t0), par, margin, s);
    if (st != PISA_OK) return st;
  }
  return PISA_OK;
}

int qm_select_final(const Geometry& g, const int32_t* par, const float* blk, int32_t* idx, float* margin, float* lse_out,
                    float* sel_lse, int32_t* status, cudaStream_t s) {
  qm::Args a = {};
  a.lgC = log2i(g.C); a.lgg = log2i(g.g); a.lgG = log2i(g.G);
  a.t0 = 0; a.t1 = g.N;
  a.status = status;
  return launch_qm_select_final(g, a, (long long)g.B * g.N, par, blk, idx, margin, lse_out, sel_lse, s);
}

}  // namespace pisa
