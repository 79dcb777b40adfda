// Dot products of 32 rows with a group's queries by one warp, fp32 (the exact SIMT kernels).
#pragma once

#include "pisa_common.cuh"

namespace pisa {

// Lane l gets the dots of row l.  D / V lanes share a row, 16 bytes each, so that a load touches whole rows (a lane per row
// costs a wavefront per lane and load, and those bound the kernels); a lane's partial sums of D / V rows are then exchanged
// so that every lane ends up with one row (D / V - 1 shuffles per head).  The sums associate the same way for every row.
template <typename T, int D, int G>
struct RowDots {
  static constexpr int V = Elem<T>::kVec, LPR = D / V;
  float q[G][V];                              // this lane's part of the queries

  __device__ __forceinline__ void load(const float* qf) {        // qf: [G][D] in shared memory
    const int sub = (threadIdx.x & 31) % LPR;
#pragma unroll
    for (int hh = 0; hh < G; ++hh)
#pragma unroll
      for (int e = 0; e < V; ++e) q[hh][e] = qf[hh * D + sub * V + e];
  }
  // rows base, base + stride, ...; n >= 1 of them exist (the last one stands in for the others)
  __device__ __forceinline__ void dots(const T* __restrict__ base, long long stride, int n, float (&z)[G]) const {
    const int lane = threadIdx.x & 31, sub = lane % LPR, first = lane - sub;
    float part[G][LPR];
#pragma unroll
    for (int i = 0; i < LPR; ++i) {
      float x[V];
      Elem<T>::load_chunk(base + (long long)min(first + i, n - 1) * stride + sub * V, x);
#pragma unroll
      for (int hh = 0; hh < G; ++hh) {
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < V; ++e) s = fmaf(x[e], q[hh][e], s);
        part[hh][i] = s;
      }
    }
#pragma unroll
    for (int o = LPR / 2; o >= 1; o >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int hh = 0; hh < G; ++hh)
#pragma unroll
        for (int i = 0; i < o; ++i) {
          const float send = up ? part[hh][i] : part[hh][i + o], mine = up ? part[hh][i + o] : part[hh][i];
          part[hh][i] = mine + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
#pragma unroll
    for (int hh = 0; hh < G; ++hh) z[hh] = part[hh][0];
  }
};

}  // namespace pisa
