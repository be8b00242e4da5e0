// The pair update of the force kernels: packed .f32x2 arithmetic on two
// reference points for one template point.
#pragma once
#include "common.cuh"
#include "ex2_poly.cuh"

namespace scgr {

// 2^-x
__device__ __forceinline__ float ex2_neg(float x) {
  float y;
  asm("{ .reg .f32 t; neg.f32 t, %1; ex2.approx.ftz.f32 %0, t; }" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

constexpr float RSQRT_CAP = 1e18f;

// 2^-e for e >= 0 on the FP32 pipe, both lanes (Cody-Waite reduction):
// e = n + g with n = round(e), g in [-1/2, 1/2]; 2^-g from the degree-5
// minimax polynomial of ex2_poly.cuh (relative error < 2^-22 in float32),
// and 2^-n added to the exponent field.  Adding 1.5 * 2^23 rounds e to an
// integer held in the low mantissa bits: t = 1.5 * 2^23 - n, whose bit
// pattern shifted left by 23 is -n << 23 for |n| < 256.  Results below
// 2^-125.5 (e >= 125.5, including e = +inf) are 0, as the special-function
// unit's flushing ex2 gives below 2^-126.
constexpr float EX2_ROUND = 12582912.0f;  // 1.5 * 2^23
constexpr float EX2_POLY_MAX = 125.5f;
__device__ __forceinline__ u64 ex2_neg_poly2(u64 e) {
  const u64 R2 = pk2(EX2_ROUND, EX2_ROUND);
  const u64 t = sub2(R2, e);   // 1.5 * 2^23 - round(e)
  const u64 nf = sub2(t, R2);  // -round(e), exact
  const u64 g = add2(e, nf);   // e - round(e), exact
  u64 q = fma2(pk2(EX2_POLY_C5, EX2_POLY_C5), g, pk2(EX2_POLY_C4, EX2_POLY_C4));
  q = fma2(q, g, pk2(EX2_POLY_C3, EX2_POLY_C3));
  q = fma2(q, g, pk2(EX2_POLY_C2, EX2_POLY_C2));
  q = fma2(q, g, pk2(EX2_POLY_C1, EX2_POLY_C1));
  q = fma2(q, g, pk2(EX2_POLY_C0, EX2_POLY_C0));
  float t0, t1, q0, q1, e0, e1;
  upk2(t, t0, t1);
  upk2(q, q0, q1);
  upk2(e, e0, e1);
  const float r0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
  const float r1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
  return pk2(e0 < EX2_POLY_MAX ? r0 : 0.f, e1 < EX2_POLY_MAX ? r1 : 0.f);
}

// One packed pair update: reference points (j, j+1) against one template point.
// POLY (p = 2 only): the factor 2^-ep on the FP32 pipe instead of the
// special-function unit.
template <int PM, bool POLY = false>
__device__ __forceinline__ void pair2(u64 xv, u64 yv, u64 zv, u64 nv, u64 av, u64 lv, u64 mx, u64 my,
                                      u64 mz, u64 ny, u64 ah, u64 nq, u64& W, u64& Sx, u64& Sy, u64& Sz) {
  u64 d2 = add2(nv, ny);
  d2 = fma2(xv, mx, d2);
  d2 = fma2(yv, my, d2);
  d2 = fma2(zv, mz, d2);
  const u64 u = sub2(av, ah);
  const u64 ep = fma2(u, u, lv);  // u^2 - L >= 0; the weight is 2^-ep times the distance factor
  u64 w;
  if (PM == 1) {
    float e0, e1;
    upk2(ep, e0, e1);
    w = pk2(ex2_neg(e0), ex2_neg(e1));
  } else if (PM == 2) {
    float e0, e1, q0, q1;
    upk2(d2, q0, q1);
    const u64 dd = pk2(sqrt_approx(fabsf(q0)), sqrt_approx(fabsf(q1)));
    if (POLY) {
      w = mul2(ex2_neg_poly2(ep), dd);
    } else {
      upk2(ep, e0, e1);
      w = mul2(pk2(ex2_neg(e0), ex2_neg(e1)), dd);
    }
  } else if (PM == 3) {
    float e0, e1;
    upk2(ep, e0, e1);
    w = mul2(pk2(ex2_neg(e0), ex2_neg(e1)), d2);
  } else if (PM == 4) {
    // p = 2 with d = d^2 / sqrt(|d^2|): a reciprocal square root and one more
    // packed multiply (kept as a tunable alternative: on GB300 rsqrt and sqrt
    // occupy the special-function unit equally, so this form is slower).
    // The cap keeps d^2 = 0 at weight 0 (0 * inf would be NaN); a d^2 below
    // the rounding of its own terms may come out with either sign.
    float e0, e1, q0, q1;
    upk2(ep, e0, e1);
    upk2(d2, q0, q1);
    const u64 r = pk2(fminf(rsqrt_approx(fabsf(q0)), RSQRT_CAP), fminf(rsqrt_approx(fabsf(q1)), RSQRT_CAP));
    w = mul2(mul2(pk2(ex2_neg(e0), ex2_neg(e1)), d2), r);
  } else {
    float q0, q1;
    upk2(d2, q0, q1);
    const u64 t = fma2(nq, pk2(lg2_approx(fabsf(q0)), lg2_approx(fabsf(q1))), ep);  // ep - q log2 d^2
    float t0, t1;
    upk2(t, t0, t1);
    w = pk2(ex2_neg(t0), ex2_neg(t1));
  }
  W = add2(W, w);
  Sx = fma2(w, xv, Sx);
  Sy = fma2(w, yv, Sy);
  Sz = fma2(w, zv, Sz);
}

}  // namespace scgr
