// Block log-sum-exp over accumulator columns in registers, shared by the kernels that score leaf blocks from TMEM.
#pragma once

#include <math_constants.h>
#include <stdint.h>

namespace pisa {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Online log-sum-exp (base 2) over one 32-column chunk of raw fp32 logits; (m, ssum) is the running
// (max, sum of 2^(x - max)) with x = raw * sl2.  sl2 > 0, so the max commutes with the scaling.
template <int NW>
__device__ __forceinline__ void lse_chunk(const uint32_t (&rr)[NW], float sl2, float& m, float& ssum) {
  float c0 = __uint_as_float(rr[0]), c1 = __uint_as_float(rr[1]);
  float c2 = __uint_as_float(rr[2]), c3 = __uint_as_float(rr[3]);
#pragma unroll
  for (int j = 4; j < NW; j += 4) {
    c0 = fmaxf(c0, __uint_as_float(rr[j]));
    c1 = fmaxf(c1, __uint_as_float(rr[j + 1]));
    c2 = fmaxf(c2, __uint_as_float(rr[j + 2]));
    c3 = fmaxf(c3, __uint_as_float(rr[j + 3]));
  }
  const float mn = fmaxf(m, fmaxf(fmaxf(c0, c1), fmaxf(c2, c3)) * sl2);
  const float neg = -mn;
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
  for (int j = 0; j < NW; j += 4) {
    a0 += ex2_approx(fmaf(__uint_as_float(rr[j]), sl2, neg));
    a1 += ex2_approx(fmaf(__uint_as_float(rr[j + 1]), sl2, neg));
    a2 += ex2_approx(fmaf(__uint_as_float(rr[j + 2]), sl2, neg));
    a3 += ex2_approx(fmaf(__uint_as_float(rr[j + 3]), sl2, neg));
  }
  ssum = ssum * ex2_approx(m - mn) + ((a0 + a1) + (a2 + a3));
  m = mn;
}
// the same with only the first `nvalid` (>= 1) columns of the chunk taking part.  The sums associate
// exactly as in lse_chunk (four interleaved accumulators), so a full row gives bit-identical results on
// either path: which path a row takes depends on the other rows of its tile, and the composition of a
// tile (the order of a list's entries) varies from run to run.
template <int NW>
__device__ __forceinline__ void lse_chunk_masked(const uint32_t (&rr)[NW], int nvalid, float sl2, float& m,
                                                 float& ssum) {
  float cm = -CUDART_INF_F;
#pragma unroll
  for (int j = 0; j < NW; ++j)
    if (j < nvalid) cm = fmaxf(cm, __uint_as_float(rr[j]));
  const float mn = fmaxf(m, cm * sl2);
  const float neg = -mn;
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int j = 0; j < NW; ++j)
    if (j < nvalid) acc[j & 3] += ex2_approx(fmaf(__uint_as_float(rr[j]), sl2, neg));
  ssum = ssum * ex2_approx(m - mn) + ((acc[0] + acc[1]) + (acc[2] + acc[3]));
  m = mn;
}

}  // namespace pisa
