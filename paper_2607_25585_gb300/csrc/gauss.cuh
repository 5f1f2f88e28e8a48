// Box-Muller for complex64 start vectors: one complex Gaussian from 2 x 53
// random bits, as the FP64 values (log, sincospi) rounded to FP32.
//
// In FP64 a value takes about 100 FP64 operations, and the FP64 pipe does 2 a
// clock and SM: 5.3 ms for 2^25 values, 99 % of the kernel.  Here every quantity
// is an unevaluated sum of two floats (Dekker, Knuth: error-free sums, products
// by FMA), carried only where the result needs it:
//   -2 ln u = -2 (e ln 2 + ln m), m in [sqrt(1/2), sqrt 2), ln m = 2 artanh((m - 1)/(m + 1)) by its series;
//   sin, cos of 2 pi f, |f| <= 1/8 turn after an exact reduction in integers, by their Taylor series.
// The coefficients whose terms exceed 1e-5 of the result are two floats, the
// series end below 1e-13: the largest relative error of a product over 4e8 values
// is 1.6e-12.  rounded() then tells whether everything within kGaussError of the
// value rounds to the same FP32 number; if not (1 value in 10^4), the FP64
// functions decide (Ziv's strategy).  So the bits are those of the FP64 form:
// start blocks of 2^20 x 32 values 4.71 -> 0.62 ms, the same bits.
#pragma once

#include <cuda_runtime.h>

namespace ftlm {

struct Two {  // hi + lo, |lo| at most a few ulp of hi (sums and products are not renormalised)
  float hi, lo;
};

__host__ __device__ __forceinline__ Two fast_two_sum(float a, float b) {  // |a| >= |b| or a = 0
  const float s = a + b;
  return {s, b - (s - a)};
}
__host__ __device__ __forceinline__ Two two_sum(float a, float b) {
  const float s = a + b, t = s - a;
  return {s, (a - (s - t)) + (b - t)};
}
__host__ __device__ __forceinline__ Two two_mul(Two a, Two b) {
#ifdef __CUDA_ARCH__
  const float p = __fmul_rn(a.hi, b.hi);  // (not contracted into the sum below)
#else
  const float p = a.hi * b.hi;
#endif
  return {p, fmaf(a.hi, b.hi, -p) + fmaf(a.hi, b.lo, a.lo * b.hi)};
}
// |a| >= |b| or a = 0
__host__ __device__ __forceinline__ Two add_smaller(Two a, Two b) {
  const Two s = fast_two_sum(a.hi, b.hi);
  return {s.hi, s.lo + (a.lo + b.lo)};
}

#define TWO(x) (Two{(float)(x), (float)((x) - (double)(float)(x))})  // a constant as two floats

__host__ __device__ __forceinline__ float approx_rcp(float x) {
#ifdef __CUDA_ARCH__
  return __frcp_rn(x);
#else
  return 1.0f / x;
#endif
}
__host__ __device__ __forceinline__ float approx_rsqrt(float x) {
#ifdef __CUDA_ARCH__
  return rsqrtf(x);
#else
  return 1.0f / sqrtf(x);
#endif
}
__host__ __device__ __forceinline__ int leading_zeros(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return __builtin_clzll(x);
#endif
}

// sqrt(-2 ln(k / 2^53)), 1 <= k <= 2^53
__host__ __device__ __forceinline__ Two box_muller_radius(unsigned long long k) {
  const int lz = leading_zeros(k);
  const unsigned long long nk = k << lz;  // k / 2^53 = (nk / 2^63) 2^e
  int e = 10 - lz;
  // a = m - 1 exactly as an integer / 2^63, or -integer / 2^64 where m = nk / 2^64 (above sqrt 2 / 2)
  const bool half = nk > 0xb504f333f9de6484ull;
  const unsigned long long ia = half ? 0ull - nk : nk - (1ull << 63);
  const float unit = half ? -0x1p-64f : 0x1p-63f;
  e += half;
  Two a = fast_two_sum((float)(unsigned)(ia >> 40) * 0x1p40f, (float)(unsigned)((ia >> 16) & 0xffffffu) * 0x1p16f);
  a = fast_two_sum(a.hi, a.lo + (float)(unsigned)(ia & 0xffffu));
  a.hi *= unit;
  a.lo *= unit;
  // s = (m - 1) / (m + 1)
  const Two b0 = two_sum(2.0f, a.hi);
  const float bl = b0.lo + a.lo, rb = approx_rcp(b0.hi);
  const float sh = a.hi * rb;
  const float rem = fmaf(-sh, b0.hi, a.hi) + (a.lo - sh * bl);
  const Two s = fast_two_sum(sh, rem * rb);
  // artanh s = s (1 + s^2 (1/3 + s^2 (1/5 + ...)))
  const Two t = two_mul(s, s);
  float q = 1.0f / 17.0f;
  q = fmaf(q, t.hi, 1.0f / 15.0f);
  q = fmaf(q, t.hi, 1.0f / 13.0f);
  q = fmaf(q, t.hi, 1.0f / 11.0f);
  q = fmaf(q, t.hi, 1.0f / 9.0f);
  q = fmaf(q, t.hi, 1.0f / 7.0f);
  const Two c = two_mul(t, add_smaller(TWO(1.0 / 3.0), two_mul(t, add_smaller(TWO(1.0 / 5.0), {q * t.hi, 0.0f}))));
  const Two sc = two_mul(s, c);
  const Two ln_m2 = add_smaller(s, sc);  // ln m / 2
  // -2 ln u = -4 (e ln(2)/2 + ln(m)/2); ln(2)/2 = 0x1.62e4p-2 (14 bits: its multiples of |e| <= 53 are exact) + rest
  const double half_ln2 = 0.34657359027997265471;
  const float l_hi = 0x1.62e4p-2f, l_lo = (float)(half_ln2 - 0x1.62e4p-2);
  const float fe = (float)e;
  const Two big = fast_two_sum(fe * l_hi, fe * l_lo);
  const Two low = {fmaf(fe, l_lo, -(fe * l_lo)), 0.0f};
  Two L = add_smaller(big, ln_m2);
  L.lo += low.hi;
  const float h = -4.0f * L.hi, l = -4.0f * L.lo;
  if (!(h > 0.0f)) return {0.0f, 0.0f};  // u = 1
  const float y = approx_rsqrt(h), r = h * y;
  return fast_two_sum(r, 0.5f * y * (fmaf(-r, r, h) + l));
}

// cos and sin of 2 pi k / 2^53, 1 <= k <= 2^53
__host__ __device__ __forceinline__ void box_muller_angle(unsigned long long k, Two& cs, Two& sn) {
  const int quad = (int)((k + (1ull << 50)) >> 51);              // nearest quarter turn
  const long long f = (long long)k - ((long long)quad << 51);    // |f| <= 2^50: f / 2^53 turns from it
  const unsigned long long m = (unsigned long long)(f < 0 ? -f : f);
  Two turn = fast_two_sum((float)(unsigned)(m >> 27) * 0x1p27f, (float)((unsigned)(m >> 3) & 0xffffffu) * 8.0f);
  turn = fast_two_sum(turn.hi, turn.lo + (float)((unsigned)m & 7u));
  const float unit = f < 0 ? -0x1p-53f : 0x1p-53f;
  const float tau = 6.283185307179586f;
  const Two th = two_mul({turn.hi * unit, turn.lo * unit}, {tau, (float)(6.283185307179586477 - (double)tau)});
  const Two u = two_mul(th, th);
  // sin th = th + th u (-1/6 + u (1/120 + u (-1/5040 + ...)))
  float p = fmaf(u.hi, 1.0f / 6227020800.0f, -1.0f / 39916800.0f);
  p = fmaf(u.hi, p, 1.0f / 362880.0f);
  Two w = add_smaller(TWO(-1.0 / 5040.0), {u.hi * p, 0.0f});
  w = add_smaller(TWO(1.0 / 120.0), two_mul(u, w));
  w = add_smaller(TWO(-1.0 / 6.0), two_mul(u, w));
  const Two s = add_smaller(th, two_mul(th, two_mul(u, w)));
  // cos th = 1 + u (-1/2 + u (1/24 + u (-1/720 + ...)))
  p = fmaf(u.hi, -1.0f / 87178291200.0f, 1.0f / 479001600.0f);
  p = fmaf(u.hi, p, -1.0f / 3628800.0f);
  p = fmaf(u.hi, p, 1.0f / 40320.0f);
  w = add_smaller(TWO(-1.0 / 720.0), {u.hi * p, 0.0f});
  w = add_smaller(TWO(1.0 / 24.0), two_mul(u, w));
  w = add_smaller({-0.5f, 0.0f}, two_mul(u, w));
  const Two c = add_smaller({1.0f, 0.0f}, two_mul(u, w));
  const bool swap = quad & 1;
  const bool negc = (quad + 1) & 2, negs = quad & 2;
  cs = swap ? s : c;
  sn = swap ? c : s;
  if (negc) cs = {-cs.hi, -cs.lo};
  if (negs) sn = {-sn.hi, -sn.lo};
}

// bound of the relative error of a product of a radius and a cosine or sine
constexpr float kGaussError = 0x1p-38f;

// a b rounded to FP32; false where the error may decide the rounding, or the product is zero
__host__ __device__ __forceinline__ bool rounded(Two a, Two b, float& out) {
  const Two p = two_mul(a, b);
  const float d = p.hi * kGaussError;
  out = p.hi + (p.lo + d);
  return out == p.hi + (p.lo - d) && p.hi != 0.0f;
}
#undef TWO

}  // namespace ftlm
