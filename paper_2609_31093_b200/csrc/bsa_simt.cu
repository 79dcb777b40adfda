// Block-sparse attention over the selected leaf blocks, exact-fp32 SIMT path
// (Eq. "selected sparse attention"; causal mask inside selected blocks, App. B).
//
// WPT warps per (b, KV head, query token) serve the G query heads of the group together, since they
// share one block set (Sec. 3.3).  Scores: one lane per key; P.V: one lane per slice of d.  Online
// softmax over chunks of 32 keys, dealt out to the token's warps, whose sums are merged at the end.
//
// Bound by the wavefronts and the latency of a warp's loads: key rows are read by several lanes each (simt_dot.cuh; not for
// large groups), value rows eight at a time, and where the tokens alone do not fill the GPU each gets four or eight warps;
// the sixteen warps of a CTA serve neighbouring tokens then, which find one another's rows in L1.  1024 tokens, one head, d = 64, four
// blocks of 64: a lane per key and one value row at a time 49 us; four warps per token and eight rows 34.
#include <math_constants.h>

#include "launch.cuh"
#include "pisa_common.cuh"
#include "simt_dot.cuh"

namespace pisa {

namespace {

template <typename T, int D, int G>
__device__ __forceinline__ void dot_row(const T* __restrict__ row, const float* __restrict__ qf,
                                        float (&z)[G]) {
  constexpr int V = Elem<T>::kVec;
#pragma unroll
  for (int h = 0; h < G; ++h) z[h] = 0.f;
#pragma unroll 2
  for (int c = 0; c < D / V; ++c) {
    float x[V];
    Elem<T>::load_chunk(row + c * V, x);
#pragma unroll
    for (int h = 0; h < G; ++h) {
      const float4* qq = reinterpret_cast<const float4*>(qf + h * D + c * V);
#pragma unroll
      for (int v4 = 0; v4 < V / 4; ++v4) {
        const float4 a = qq[v4];
        z[h] = fmaf(x[4 * v4 + 0], a.x, z[h]);
        z[h] = fmaf(x[4 * v4 + 1], a.y, z[h]);
        z[h] = fmaf(x[4 * v4 + 2], a.z, z[h]);
        z[h] = fmaf(x[4 * v4 + 3], a.w, z[h]);
      }
    }
  }
}
}  // namespace

template <typename T, int D, int G, int WPT>
__global__ void __launch_bounds__(WPT == 1 ? 128 : 512)
bsa_simt_kernel(Geometry geo, const T* __restrict__ q, const T* __restrict__ k, const T* __restrict__ v,
                const int32_t* __restrict__ idx, T* __restrict__ out, float* __restrict__ lse) {
  constexpr int DV = D / 32;                  // output dims per lane
  constexpr int TPC = WPT == 1 ? 4 : 16 / WPT;   // tokens per CTA
  constexpr int UV = G <= 4 ? 8 : 4;          // value rows in flight
  __shared__ __align__(16) float s_q[TPC][G * D];
  __shared__ float s_acc[WPT > 1 ? TPC : 1][WPT > 1 ? WPT : 1][WPT > 1 ? G * D : 1], s_ml[WPT > 1 ? TPC : 1][WPT > 1 ? WPT : 1][2 * G];
  const int lane = threadIdx.x & 31, tok = (threadIdx.x >> 5) / WPT, part = (threadIdx.x >> 5) % WPT;
  const int gtid = part * 32 + lane;          // thread of the token's group
  auto group_sync = [&]() {
    if (WPT == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + tok), "r"(WPT * 32) : "memory");
  };
  grid_dependency();
  const long long w = (long long)blockIdx.x * TPC + tok;
  const long long total = (long long)geo.B * geo.Hkv * geo.N;
  if (w >= total) return;
  const int t = (int)(w % geo.N);
  const int h = (int)((w / geo.N) % geo.Hkv);
  const int b = (int)(w / ((long long)geo.N * geo.Hkv));

  float* qf = s_q[tok];
  for (int hh = 0; hh < G; ++hh) {
    const T* row = q + (long long)b * geo.qs[0] + (long long)t * geo.qs[1] + (long long)(h * G + hh) * geo.qs[2];
    for (int e = gtid; e < D; e += WPT * 32) qf[hh * D + e] = Elem<T>::to_float(row[e]);
  }
  group_sync();

  RowDots<T, D, G <= 2 ? G : 1> rows;
  if constexpr (G <= 2) rows.load(qf);
  float acc[G][DV];
  float m[G], l[G];
#pragma unroll
  for (int hh = 0; hh < G; ++hh) {
    m[hh] = -CUDART_INF_F; l[hh] = 0.f;
#pragma unroll
    for (int e = 0; e < DV; ++e) acc[hh][e] = 0.f;
  }
  const T* kb = k + (long long)b * geo.ks[0] + (long long)h * geo.ks[2];
  const T* vb = v + (long long)b * geo.vs[0] + (long long)h * geo.vs[2];
  const int32_t* sel = idx + w * (long long)geo.K;

  int chunk = 0, blks = -1;
  for (int slot = 0; slot < geo.K; ++slot) {
    if ((slot & 31) == 0) blks = slot + lane < geo.K ? sel[slot + lane] : -1;
    const int blk = __shfl_sync(0xffffffffu, blks, slot & 31);
    if (blk < 0 || blk >= geo.M[1]) continue;
    const int lo = blk * geo.C;
    const int hi = min(min(lo + geo.C, geo.N), t + 1);     // causal: keys j <= t only
    for (int j0 = lo; j0 < hi; j0 += 32) {
      if (WPT > 1 && chunk++ % WPT != part) continue;
      const int j = j0 + lane;
      const bool valid = j < hi;
      float z[G], p[G];
      if constexpr (G <= 2) {
        rows.dots(kb + (long long)j0 * geo.ks[1], geo.ks[1], hi - j0, z);
      } else if (valid) {
        dot_row<T, D, G>(kb + (long long)j * geo.ks[1], qf, z);
      } else {
#pragma unroll
        for (int hh = 0; hh < G; ++hh) z[hh] = 0.f;
      }
#pragma unroll
      for (int hh = 0; hh < G; ++hh) {
        const float zz = valid ? z[hh] * geo.scale : -CUDART_INF_F;
        const float mn = fmaxf(m[hh], warp_max(zz));
        p[hh] = valid ? expf(zz - mn) : 0.f;
        const float alpha = expf(m[hh] - mn);
        l[hh] = l[hh] * alpha + warp_sum(p[hh]);
#pragma unroll
        for (int e = 0; e < DV; ++e) acc[hh][e] *= alpha;
        m[hh] = mn;
      }
      const int cnt = min(32, hi - j0);
      for (int jj = 0; jj < cnt; jj += UV) {
        float xv[UV][DV];
#pragma unroll
        for (int u = 0; u < UV; ++u) {
          const T* vr = vb + (long long)(j0 + min(jj + u, cnt - 1)) * geo.vs[1] + lane * DV;
          if constexpr (DV == 2 && sizeof(T) == 4) {
            const float2 x = *reinterpret_cast<const float2*>(vr);
            xv[u][0] = x.x;
            xv[u][DV - 1] = x.y;
          } else if constexpr (DV == 4 && sizeof(T) == 4) {
            const float4 x = *reinterpret_cast<const float4*>(vr);
            xv[u][0] = x.x; xv[u][DV - 3] = x.y; xv[u][DV - 2] = x.z; xv[u][DV - 1] = x.w;
          } else {
#pragma unroll
            for (int e = 0; e < DV; ++e) xv[u][e] = Elem<T>::to_float(vr[e]);
          }
        }
#pragma unroll
        for (int u = 0; u < UV; ++u) {
          if (jj + u >= cnt) break;
#pragma unroll
          for (int hh = 0; hh < G; ++hh) {
            const float ph = __shfl_sync(0xffffffffu, p[hh], jj + u);
#pragma unroll
            for (int e = 0; e < DV; ++e) acc[hh][e] = fmaf(ph, xv[u][e], acc[hh][e]);
          }
        }
      }
    }
  }
  if constexpr (WPT > 1) {
#pragma unroll
    for (int hh = 0; hh < G; ++hh) {
#pragma unroll
      for (int e = 0; e < DV; ++e) s_acc[tok][part][hh * D + lane * DV + e] = acc[hh][e];
      if (lane == 0) { s_ml[tok][part][2 * hh] = m[hh]; s_ml[tok][part][2 * hh + 1] = l[hh]; }
    }
    group_sync();
    for (int x = gtid; x < G * D; x += WPT * 32) {
      const int hh = x / D, hq = h * G + hh;
      float mx = -CUDART_INF_F, sum = 0.f, o = 0.f;
#pragma unroll
      for (int p = 0; p < WPT; ++p) mx = fmaxf(mx, s_ml[tok][p][2 * hh]);
#pragma unroll
      for (int p = 0; p < WPT; ++p) {
        const float lp = s_ml[tok][p][2 * hh + 1], f = lp != 0.f ? expf(s_ml[tok][p][2 * hh] - mx) : 0.f;   // (a warp without keys: m = -inf; a NaN stays)
        sum = fmaf(lp, f, sum);
        o = fmaf(s_acc[tok][p][x], f, o);
      }
      out[(long long)b * geo.os[0] + (long long)t * geo.os[1] + (long long)hq * geo.os[2] + x - hh * D] = Elem<T>::from_float(sum != 0.f ? o / sum : 0.f);
      if (x == hh * D) lse[((long long)b * geo.Hq + hq) * geo.N + t] = sum > 0.f ? mx + logf(sum) : -CUDART_INF_F;
    }
    return;
  }
#pragma unroll
  for (int hh = 0; hh < G; ++hh) {
    const int hq = h * G + hh;
    const float inv = (l[hh] > 0.f) ? 1.f / l[hh] : 0.f;
    T* orow = out + (long long)b * geo.os[0] + (long long)t * geo.os[1] + (long long)hq * geo.os[2] + lane * DV;
#pragma unroll
    for (int e = 0; e < DV; ++e) orow[e] = Elem<T>::from_float(acc[hh][e] * inv);
    if (lane == 0)
      lse[((long long)b * geo.Hq + hq) * geo.N + t] = (l[hh] > 0.f) ? m[hh] + logf(l[hh]) : -CUDART_INF_F;
  }
}

template <typename T, int D, int G>
static int launch_tdg(const Geometry& g, const void* q, const void* k, const void* v, const int32_t* idx,
                      void* out, float* lse, cudaStream_t s) {
  const long long total = (long long)g.B * g.Hkv * g.N;
  const long long ctas = (total + 3) / 4;
  if (ctas > 0x7fffffffLL) return PISA_ERR_UNSUPPORTED;
  // four warps per token while that leaves no SM with more than its 64, eight below a third of that (larger groups have work for
  // a warp's loads to hide behind).  One head, d = 64: 300 tokens 36.7 us with four, 28.8 with eight (whole forward, the routing
  // split alike), 600 tokens 44.7 and 41.2, 1024 tokens 47.0 and 53.9
  if constexpr (G <= 2) {
    if (total <= 5LL * num_sms())
      return launch_dependent<bsa_simt_kernel<T, D, G, 8>>("bsa_simt", dim3((unsigned)((total + 1) / 2)), 512u, 0, s, g, (const T*)q,
                                                           (const T*)k, (const T*)v, idx, (T*)out, lse);
    if (total <= 16LL * num_sms()) {
      return launch_dependent<bsa_simt_kernel<T, D, G, 4>>("bsa_simt", dim3((unsigned)ctas), 512u, 0, s, g, (const T*)q, (const T*)k,
                                                           (const T*)v, idx, (T*)out, lse);
    }
  }
  return launch_dependent<bsa_simt_kernel<T, D, G, 1>>("bsa_simt", dim3((unsigned)ctas), 128u, 0, s, g, (const T*)q, (const T*)k,
                                                       (const T*)v, idx, (T*)out, lse);
}

template <typename T, int D>
static int launch_td(const Geometry& g, const void* q, const void* k, const void* v, const int32_t* idx,
                     void* out, float* lse, cudaStream_t s) {
  switch (g.G) {
    case 1: return launch_tdg<T, D, 1>(g, q, k, v, idx, out, lse, s);
    case 2: return launch_tdg<T, D, 2>(g, q, k, v, idx, out, lse, s);
    case 4: return launch_tdg<T, D, 4>(g, q, k, v, idx, out, lse, s);
    case 8: return launch_tdg<T, D, 8>(g, q, k, v, idx, out, lse, s);
    case 16: return launch_tdg<T, D, 16>(g, q, k, v, idx, out, lse, s);
    default: return PISA_ERR_UNSUPPORTED;
  }
}

template <typename T>
static int launch_t(const Geometry& g, const void* q, const void* k, const void* v, const int32_t* idx,
                    void* out, float* lse, cudaStream_t s) {
  switch (g.d) {
    case 32: return launch_td<T, 32>(g, q, k, v, idx, out, lse, s);
    case 64: return launch_td<T, 64>(g, q, k, v, idx, out, lse, s);
    case 128: return launch_td<T, 128>(g, q, k, v, idx, out, lse, s);
    default: return PISA_ERR_UNSUPPORTED;
  }
}

int launch_bsa_simt(const Geometry& g, int dtype, const void* q, const void* k, const void* v,
                    const int32_t* idx, void* out, float* lse, cudaStream_t s) {
  if (dtype == PISA_BF16) return launch_t<__nv_bfloat16>(g, q, k, v, idx, out, lse, s);
  return launch_t<float>(g, q, k, v, idx, out, lse, s);
}

}  // namespace pisa
