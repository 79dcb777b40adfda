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

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// two fp32 lanes in one instruction (sm_100); the same roundings as the scalar forms
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// 2^z for two z on the FMA pipe, where the special-function unit (16 exponentials per clock and SM) is the limit: z = n + f
// with n the nearest integer (Cody and Waite), a polynomial of degree five for 2^f on [-1/2, 1/2] with value 1 at 0 (relative
// minimax by linear programming, 1.1e-7; 1.7e-7 with its fp32 roundings, what ex2.approx states), the exponent by integer
// arithmetic.  z < -126 counts as -126; z < 128.
__device__ __forceinline__ float max_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ uint64_t exp2_fma2(float z0, float z1) {
  const uint64_t z = pack2(max_nan(z0, -126.f), max_nan(z1, -126.f));
  const uint64_t r = add2(z, pack2(12582912.f, 12582912.f));        // 1.5 * 2^23: n in the low bits
  const uint64_t f = fma2(add2(r, pack2(-12582912.f, -12582912.f)), pack2(-1.f, -1.f), z);
  uint64_t p = fma2(f, pack2(0.001326472731307149f, 0.001326472731307149f), pack2(0.009671512991189957f, 0.009671512991189957f));
  p = fma2(f, p, pack2(0.05550733581185341f, 0.05550733581185341f));
  p = fma2(f, p, pack2(0.24022242426872253f, 0.24022242426872253f));
  p = fma2(f, p, pack2(0.6931470036506653f, 0.6931470036506653f));
  p = fma2(f, p, pack2(1.f, 1.f));
  float r0, r1;
  unpack2(r, r0, r1);
  constexpr int one = 127 << 23;                                    // bits of 1.0f
  return mul2(p, pack2(__int_as_float((__float_as_int(r0) << 23) + one), __int_as_float((__float_as_int(r1) << 23) + one)));
}
// spreads `poly` of every eight pairs evenly
__device__ __forceinline__ constexpr bool exp_poly_pair(int pair, int poly) { return (pair % 8 + 1) * poly / 8 > (pair % 8) * poly / 8; }

// Online log-sum-exp (base 2) over one 32-column chunk of raw fp32 logits; (m, ssum) is the running
// (max, sum of 2^(x - max)) with x = raw * sl2.  sl2 > 0, so the max commutes with the scaling.
// POLY: of every eight pairs of columns, how many exponentials take the FMA pipe.
template <int NW, int POLY = 0>
__device__ __forceinline__ void lse_chunk(const uint32_t (&rr)[NW], float sl2, float& m, float& ssum) {
  float c0 = __uint_as_float(rr[0]), c1 = __uint_as_float(rr[1]);
#pragma unroll
  for (int j = 2; j < NW - 2; j += 4) {
    c0 = max3(c0, __uint_as_float(rr[j]), __uint_as_float(rr[j + 1]));
    c1 = max3(c1, __uint_as_float(rr[j + 2]), __uint_as_float(rr[j + 3]));
  }
  c0 = max3(c0, __uint_as_float(rr[NW - 2]), __uint_as_float(rr[NW - 1]));
  const float mn = fmaxf(m, fmaxf(c0, c1) * sl2);
  const uint64_t neg = pack2(-mn, -mn), sc = pack2(sl2, sl2);
  uint64_t a01 = pack2(0.f, 0.f), a23 = a01;
#pragma unroll
  for (int j = 0; j < NW; j += 4) {
    float x0, x1, x2, x3;
    unpack2(fma2(pack2(__uint_as_float(rr[j]), __uint_as_float(rr[j + 1])), sc, neg), x0, x1);
    unpack2(fma2(pack2(__uint_as_float(rr[j + 2]), __uint_as_float(rr[j + 3])), sc, neg), x2, x3);
    a01 = add2(a01, exp_poly_pair(j / 2, POLY) ? exp2_fma2(x0, x1) : pack2(ex2_approx(x0), ex2_approx(x1)));
    a23 = add2(a23, exp_poly_pair(j / 2 + 1, POLY) ? exp2_fma2(x2, x3) : pack2(ex2_approx(x2), ex2_approx(x3)));
  }
  float a0, a1, a2, a3;
  unpack2(a01, a0, a1);
  unpack2(a23, a2, a3);
  ssum = ssum * ex2_approx(m - mn) + ((a0 + a1) + (a2 + a3));
  m = mn;
}
// the same with only the first `nvalid` (>= 1) columns of the chunk taking part.  The sums associate
// exactly as in lse_chunk (four interleaved accumulators), so a full row gives bit-identical results on
// either path where lse_chunk takes no polynomial (POLY = 0, the list-driven kernels): which path a row takes depends on the other rows of its tile, and the composition of a
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
