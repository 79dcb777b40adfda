// Host side of the decoding step (the kernel and its description: decode_kernel.cuh).
#include "decode_kernel.cuh"

namespace pisa {

bool decode_supported(const Geometry& g, int dtype) {
  return dtype == PISA_BF16 && (g.d == 64 || g.d == 128) && g.G <= 16 &&
         (g.C == 64 || g.C == 128 || g.C == 32) && (long long)g.B * g.Hkv <= 65535;
}

// (the kernel keeps its partials on chip: nothing but the status word is needed)
size_t decode_workspace_bytes(const Geometry& g) { (void)g; return 0; }

int launch_decode_step(const Geometry& g, int pos, const void* q, const void* k, const void* v, void* pyramid,
                       int32_t* idx, void* out, float* lse, void* ws, cudaStream_t s) {
  (void)ws;
  DecArgs a;
  a.pos = pos;
  a.units = g.B * g.Hkv;
  a.q = (const __nv_bfloat16*)q; a.k = (const __nv_bfloat16*)k; a.v = (const __nv_bfloat16*)v;
  a.pyr = (__nv_bfloat16*)pyramid; a.idx = idx; a.out = (__nv_bfloat16*)out; a.lse = lse;
  // the path's nodes per level, and where the walk starts: the highest level with more than K live nodes
  const int c = pos / g.C;
  for (int l = 0; l < kMaxLevels; ++l) a.anc[l] = a.prev[l] = a.tile0[l] = 0;
  for (int l = 1; l <= g.L; ++l) {
    a.anc[l] = (int)(c / g.span[l]);
    a.prev[l] = (c >= 1) ? (int)((c - 1) / g.span[l]) : 0;
  }
  a.l_top = 1;
  for (int l = g.L; l >= 2; --l)
    if (a.anc[l] + 1 > g.K) { a.l_top = l; break; }
  a.n_init = 1;                                             // the root, when the walk starts there
  if (a.l_top < g.L) {
    const long long n = (long long)(a.anc[a.l_top + 1] + 1) * g.g;
    a.n_init = (int)(n < g.M[a.l_top] ? n : g.M[a.l_top]);
  }
  // the up-front scoring: every live node of the levels that can prune, in rounds of eight, when its table holds them all
  a.n_tiles = 0;
  long long tiles = 0;
  for (int l = 2; l <= a.l_top; ++l) {
    a.tile0[l] = (int)tiles;
    tiles += (a.anc[l] + 7) / 8;
    if (tiles * 8 > kDecTabNodes) break;
  }
  if (tiles * 8 <= kDecTabNodes) a.n_tiles = (int)tiles;
  if (g.d == 128) return launch_decode_d128(g, a, s);
  if (g.d == 64) return launch_decode_d64(g, a, s);
  return PISA_ERR_UNSUPPORTED;
}

}  // namespace pisa
