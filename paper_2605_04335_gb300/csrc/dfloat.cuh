// Double-FP32 outer loop of the mixed-precision solve (precision mode 2).
//
// Iterative refinement needs the fine residual r = b - lambda - A p in a precision well
// above that of the inner FP32 multigrid; the classical three-precision choice is a
// residual precision equal to the square of the inner one (2^-48 for FP32).  GB300 issues
// FP64 at about 1/64 of its FP32 rate, so native FP64 makes the residual the most
// expensive kernel of a refinement step.  This mode keeps the accumulated solution p, the
// right-hand side b and the stencil coefficients as unevaluated sums hi + lo of two floats
// (48 significant bits) and forms the residual with error-free transformations on the
// FP32 pipe:
//   two_sum(a, b)       s + e = a + b exactly                 (Knuth, 6 flops)
//   fast_two_sum(a, b)  s + e = a + b exactly when |a| >= |b|  (Dekker, 3 flops)
//   two_prod(a, b)      p + e = a * b exactly                  (one FMA for e)
// A product of two pairs keeps hi*hi exactly plus the two cross terms (dropping lo*lo,
// 2^-48 relative); the seven stencil products and b - lambda are summed with two_sum on
// the high parts and a plain float sum of all low parts.  The residual then carries an
// error of a few units of 2^-48 times sum |c| |p| over the stencil, the same form as the
// FP64 residual's 2^-53 bound.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace ibm {
namespace dfl {

__device__ __forceinline__ void two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

__device__ __forceinline__ void fast_two_sum(float a, float b, float &s, float &e) {
  s = a + b;
  e = b - (s - a);
}

// (acc_h, acc_l) += (a_h, a_l) * (b_h, b_l); acc_l collects every low-order part
__device__ __forceinline__ void acc_prod(float ah, float al, float bh, float bl, float &acc_h, float &acc_l) {
  const float p = ah * bh;
  float e = fmaf(ah, bh, -p);
  e = fmaf(ah, bl, e);
  e = fmaf(al, bh, e);
  float s, t;
  two_sum(acc_h, p, s, t);
  acc_h = s;
  acc_l += t + e;
}

// Two cells' floats side by side: sm_103a's packed FP32 operations, each component rounded as the
// scalar operation, at half the instructions.
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float x, float y) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void un2(F2 a, float &x, float &y) { asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v)); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 neg2(F2 a) { return F2{a.v ^ 0x8000000080000000ull}; }

// (acc_h, acc_l) -= (c, c_l) * (b_h, b_l): the bits of acc_prod(-c, -c_l, ...); n, nl: -c and -c_l
__device__ __forceinline__ void acc_prod_neg2(F2 c, F2 n, F2 nl, F2 bh, F2 bl, F2 &acc_h, F2 &acc_l) {
  const F2 p = mul2(c, bh);
  F2 e = fma2(n, bh, p);   // -(c b - p)
  e = fma2(n, bl, e);
  e = fma2(nl, bh, e);
  const F2 s = sub2(acc_h, p), bb = sub2(s, acc_h);
  const F2 t = sub2(sub2(acc_h, sub2(s, bb)), add2(p, bb));
  acc_h = s;
  acc_l = add2(acc_l, add2(t, e));
}
// (acc_h, acc_l) += (d, d_l) * (b_h, b_l)
__device__ __forceinline__ void acc_prod2(F2 d, F2 dl, F2 bh, F2 bl, F2 &acc_h, F2 &acc_l) {
  const F2 p = mul2(d, bh);
  F2 e = fma2(d, bh, neg2(p));
  e = fma2(d, bl, e);
  e = fma2(dl, bh, e);
  const F2 s = add2(acc_h, p), bb = sub2(s, acc_h);
  const F2 t = add2(sub2(acc_h, sub2(s, bb)), sub2(p, bb));
  acc_h = s;
  acc_l = add2(acc_l, add2(t, e));
}
__device__ __forceinline__ void two_sum2(F2 a, F2 b, F2 &s, F2 &e) {
  s = add2(a, b);
  const F2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}

// exact float -> double widening by bit manipulation (keeps the FP64 pipe free); normal
// floats, zero and inf map exactly, NaN to a NaN; subnormal floats (below 2^-126, far under any
// low part that matters here) become signed zero
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x);
  const uint32_t s = u & 0x80000000u, ex = (u >> 23) & 0xffu, m = u & 0x7fffffu;
  uint32_t hi, lo = m << 29;
  if (ex == 0) hi = s, lo = 0u;
  else if (ex == 0xffu) hi = s | 0x7ff00000u | (m ? 0x80000u : 0u);   // inf, or a quiet NaN
  else hi = s | ((ex + 896u) << 20) | (m >> 3);
  return __hiloint2double((int)hi, (int)lo);
}

// double -> float by truncating the significand (bit manipulation after the IEEE 754
// binary64 / binary32 layouts, so the FP64 pipe stays free): normal results lie within one
// unit in the last place of the float, toward zero; magnitudes below 2^-126 become signed
// zero, above the float range infinity, and a NaN stays a NaN
__device__ __forceinline__ float narrow_trunc(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t s = hi & 0x80000000u, ex = (hi >> 20) & 0x7ffu;
  uint32_t bits;
  if (ex <= 896u) bits = s;
  else if (ex >= 1151u) bits = s | 0x7f800000u | ((ex == 0x7ffu && ((hi & 0xfffffu) | lo)) ? 0x400000u : 0u);
  else bits = s | ((ex - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
  return __uint_as_float(bits);
}

// hi + lo as a double (one FP64 add)
__device__ __forceinline__ double join(float h, float l) { return widen(h) + widen(l); }

// double -> (hi, lo): hi the nearest float, lo the nearest float to the remainder.  The conversions
// and the difference run on the FP64 pipe (94 us to split 256^3 values, bound by it), so values whose
// parts are normal floats or zero are split on the integer pipe, to the same bits: the significand rounded
// half to even at 23 bits, the remainder an integer of at most 28 bits, converted and scaled.
__device__ __forceinline__ void split(double x, float &h, float &l) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x), m = b & 0x7fffffffffffffffull;
  const uint32_t s = (uint32_t)(b >> 32) & 0x80000000u, ex = (uint32_t)(m >> 52);
  if (m == 0ull) {
    h = __uint_as_float(s);
    l = 0.f;
  } else if (ex - 950u < 200u) {
    const unsigned long long t = (m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29;
    const int rem = (int)(long long)(m - (t << 29));
    h = __uint_as_float(s | ((uint32_t)t - (896u << 23)));
    l = (float)(s ? -rem : rem) * __uint_as_float((ex - 948u) << 23);
  } else {
    h = __double2float_rn(x);
    l = __double2float_rn(x - widen(h));
  }
}

}  // namespace dfl
}  // namespace ibm
