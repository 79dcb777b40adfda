// Host side of the query-major kernels (see query_major.cuh): what they support, when they are the better choice, their
// workspace, and the sequence of launches.
#include "pisa_tensor.cuh"
#include "query_major.cuh"

namespace pisa {

namespace {

constexpr int kDenseMaxTokens = 32768;                 // 256 steps of 128 keys: the attention kernel's step lists
constexpr size_t kDenseMaxBytes = (size_t)4 << 30;     // score tables (they grow with N * M1)

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

// Two tiles per work item halve the key / value traffic, which bounds the dense kernels, once there are enough pairs for
// four waves of one item per SM (4096 tokens x 16 heads still runs 5 % faster with one tile per item, 8192 5 % slower).
int tiles_per_item(const Geometry& g, long long unit_tokens) {
  return unit_tokens * g.G / 256 >= 4LL * num_sms() ? 2 : 1;
}

qm::Args uniform_args(const Geometry& g, char* ws, const Layout& l, int32_t* status) {
  qm::Args a = {};
  a.lgC = log2i(g.C); a.lgg = log2i(g.g); a.lgG = log2i(g.G);
  a.t0 = 0; a.t1 = g.N;
  a.tiles = tiles_per_item(g, (long long)g.B * g.Hkv * g.N);
  const int tpt = a.tiles * 128 / g.G;
  a.n_items = g.B * g.Hkv * ((g.N + tpt - 1) / tpt);
  a.want_leaf = 1;
  a.leaf = (float*)(ws + l.leaf); a.up = (float*)(ws + l.up); a.bits = (uint32_t*)(ws + l.bits);
  a.ctr = (int32_t*)(ws + l.ctr);
  a.status = status;
  return a;
}

}  // namespace

bool qm_supported(const Geometry& g, int dtype) {
  if (dtype != PISA_BF16 || g.score_mode != PISA_SCORE_LSE) return false;
  if ((g.d != 64 && g.d != 128) || (g.C != 64 && g.C != 128)) return false;
  return g.g == 2 || g.g == 4;
}

// Where the dense kernels win.  They cost a row N / 2 keys whatever it selects; the lists cost it K (token, block) pairs of
// gathered query rows and fp32 reductions, so the line lies at a length proportional to K.  Measured crossovers of the
// whole forward: 16 KV heads without groups (G = 1) beyond 32768 tokens at K = 16; G = 4, C = 64, K = 16 at 18 to 20
// thousand; G = 4, C = 128, K = 32 (larger blocks per pair) at 24 thousand; G = 16, d = 64, K = 8 at 8 thousand.
bool qm_dense_preferred(const Geometry& g, int dtype) {
  if (!qm_supported(g, dtype) || g.M[1] > 512 || g.N > kDenseMaxTokens) return false;
  const int per_block = g.G == 1 ? 2048 : (g.C == 128 ? 704 : 1024);
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
  return launch_qm_attend(g, a, q, k, v, g.N, lse, out, s);
}

}  // namespace pisa
