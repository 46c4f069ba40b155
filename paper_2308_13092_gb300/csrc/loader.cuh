// loader.cuh -- the loader's Box-Muller velocities, defined in FP64 and rounded
// to FP32, mostly without FP64 instructions.
//
// The definition is sd * (sqrt(-2 log u1) * cos(2 pi u2)) in FP64, then FP32.
// FP64 log, sine, cosine and root are some 250 instructions per particle at 1/64
// of the FP32 rate on this part.  Here the same product is formed in pairs of
// floats, with a bound on its distance from the FP64 result.  Where every value
// within the bound rounds to the same float, that is the result; the few others
// (three in 10^5) take the FP64 path.  Measured errors (1.6e8 draws against
// 80-bit arithmetic, approximate divisions and roots off by up to 2 ulp): radius
// 2^-46.0, sine and cosine 2^-45.8, product 2^-45.2; the bound takes 2^-40.  The
// series are the Taylor series of sine and cosine on |x| <= pi/4 and of 2 atanh;
// the two-float arithmetic is Dekker's.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace ecpic {
namespace {

struct Pair {  // hi + lo, |lo| <= ulp(hi) / 2
  float hi, lo;
};
__device__ __forceinline__ Pair renorm(float a, float b) {  // |a| >= |b|
  const float s = a + b;
  return {s, b - (s - a)};
}
__device__ __forceinline__ Pair two_sum(float a, float b) {
  const float s = a + b, z = s - a;
  return {s, (a - (s - z)) + (b - z)};
}
__device__ __forceinline__ Pair mul(Pair a, Pair b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  return renorm(p, e);
}
__device__ __forceinline__ Pair add(Pair a, Pair b) {
  const Pair s = two_sum(a.hi, b.hi), t = two_sum(a.lo, b.lo);
  const Pair u = renorm(s.hi, s.lo + t.hi);
  return renorm(u.hi, u.lo + t.lo);
}
#define ECPIC_PAIR(name, c) \
  const Pair name = {(float)(c), (float)((c) - (double)(float)(c))}

// an integer of up to 33 bits, exactly
__device__ __forceinline__ Pair from_int(long long v) {
  const float h = (float)v;
  return {h, (float)(v - (long long)h)};
}

// sin x / x as a series in z = x^2 <= 0.617, to 2^-46
__device__ __forceinline__ Pair sin_series(Pair z) {
  // from z^5 on a float is enough: the terms are below 2^-28
  float t = __fmaf_rn(-7.6471637e-13f, z.hi, 1.6059044e-10f);  // 1/15!, 1/13!
  t = __fmaf_rn(t, z.hi, -2.5052108e-8f);                      // 1/11!
  ECPIC_PAIR(c4, 1.0 / 362880.0);
  ECPIC_PAIR(c3, -1.0 / 5040.0);
  ECPIC_PAIR(c2, 1.0 / 120.0);
  ECPIC_PAIR(c1, -1.0 / 6.0);
  Pair p = add(c4, {t * z.hi, 0.0f});
  p = add(c3, mul(p, z));
  p = add(c2, mul(p, z));
  p = add(c1, mul(p, z));
  return add({1.0f, 0.0f}, mul(p, z));
}
__device__ __forceinline__ Pair cos_series(Pair z) {
  float t = __fmaf_rn(4.7794773e-14f, z.hi, -1.1470746e-11f);  // 1/16!, 1/14!
  t = __fmaf_rn(t, z.hi, 2.0876757e-9f);                       // 1/12!
  t = __fmaf_rn(t, z.hi, -2.7557319e-7f);                      // 1/10!
  ECPIC_PAIR(c4, 1.0 / 40320.0);
  ECPIC_PAIR(c3, -1.0 / 720.0);
  ECPIC_PAIR(c2, 1.0 / 24.0);
  Pair p = add(c4, {t * z.hi, 0.0f});
  p = add(c3, mul(p, z));
  p = add(c2, mul(p, z));
  p = add({-0.5f, 0.0f}, mul(p, z));
  return add({1.0f, 0.0f}, mul(p, z));
}

// cosine and sine of 2 pi t / 2^32
__device__ __forceinline__ void turn(uint32_t t, Pair* c, Pair* s) {
  const uint32_t k = (t + (1u << 29)) >> 30;  // nearest quarter turn
  const int d = (int)(t - (k << 30));         // -2^29 .. 2^29
  ECPIC_PAIR(quarter, 1.5707963267948966 / 1073741824.0);
  const Pair x = mul(from_int(d), quarter);
  const Pair z = mul(x, x);
  const Pair sx = mul(x, sin_series(z)), cx = cos_series(z);
  const Pair a = (k & 1u) ? sx : cx, b = (k & 1u) ? cx : sx;  // |cos|, |sin| up to signs
  const bool nc = ((k + 1u) & 2u) != 0u, ns = (k & 2u) != 0u;
  *c = {nc ? -a.hi : a.hi, nc ? -a.lo : a.lo};
  *s = {ns ? -b.hi : b.hi, ns ? -b.lo : b.lo};
}

// sqrt(-2 log(m / 2^32)) for 1 <= m < 2^32
__device__ __forceinline__ Pair radius(uint32_t m) {
  // m = 2^e w with w in [sqrt(1/2), sqrt(2))
  int e = 31 - __clz((int)(m | 1u));  // (m = 0 is a case for the caller)
  uint32_t a = m << (31 - e);  // w = a / 2^31 in [1, 2)
  long long num, den;          // (w - 1) / (w + 1)
  if (a >= 0xB504F334u) {      // w >= sqrt(2): halve it
    ++e;
    num = (long long)a - (1ll << 32);
    den = (long long)a + (1ll << 32);
  } else {
    num = (long long)a - (1ll << 31);
    den = (long long)a + (1ll << 31);
  }
  const Pair n = from_int(num), d = from_int(den);
  const float q = __fdividef(n.hi, d.hi);
  // q + (n - q d) / d, twice corrected
  float r = __fmaf_rn(-q, d.hi, n.hi);
  r = __fmaf_rn(-q, d.lo, r + n.lo);
  const float q1 = __fdividef(r, d.hi);
  const Pair s = renorm(q, q1);
  // the remainder of both parts, so that the quotient is good to 2^-46
  const Pair sd = mul(s, d);
  const float rr = ((n.hi - sd.hi) - sd.lo) + n.lo;
  const Pair s2 = add(s, {__fdividef(rr, d.hi), 0.0f});
  const Pair z = mul(s2, s2);  // <= 0.0295
  // atanh(s) / s = 1 + z/3 + z^2/5 + ...; from z^4 on a float is enough
  float t = __fmaf_rn(1.0f / 19.0f, z.hi, 1.0f / 17.0f);
  t = __fmaf_rn(t, z.hi, 1.0f / 15.0f);
  t = __fmaf_rn(t, z.hi, 1.0f / 13.0f);
  t = __fmaf_rn(t, z.hi, 1.0f / 11.0f);
  t = __fmaf_rn(t, z.hi, 1.0f / 9.0f);
  ECPIC_PAIR(c3, 1.0 / 7.0);
  ECPIC_PAIR(c2, 1.0 / 5.0);
  ECPIC_PAIR(c1, 1.0 / 3.0);
  Pair p = add(c3, {t * z.hi, 0.0f});
  p = add(c2, mul(p, z));
  p = add(c1, mul(p, z));
  p = add({1.0f, 0.0f}, mul(p, z));
  const Pair lw = mul(s2, p);  // log(w) / 2
  // -2 log(m / 2^32) = 2 (32 - e) log 2 - 4 (log(w) / 2)
  ECPIC_PAIR(ln2, 0.69314718055994531);
  const float turns = 2.0f * (float)(32 - e);
  const Pair l = add(mul({turns, 0.0f}, ln2), {-4.0f * lw.hi, -4.0f * lw.lo});
  const float y = rsqrtf(l.hi), g = l.hi * y;
  const float res = __fmaf_rn(-g, g, l.hi) + l.lo;  // l - g^2
  const Pair r1 = renorm(g, 0.5f * y * res);
  // once more: the remainder of the pair
  const Pair sq = mul(r1, r1);
  const float res2 = (l.hi - sq.hi) + (l.lo - sq.lo);
  return add(r1, {0.5f * y * res2, 0.0f});
}

// The float that sd * (r * c) rounds to, where the pair product decides it:
// the FP64 result is within 2^-40 + 2^-48 / |c| of it, relatively (2^-45 for
// the pairs, 2^-49 for FP64's own roundings but the angle's, whose 2^-49.7
// weigh 1 / |c|).  Powers of two (uneven neighbours) and tiny values are left
// to FP64.
__device__ __forceinline__ bool certain(Pair sd, Pair r, Pair c, float* out) {
  const Pair v = mul(sd, mul(r, c));
  const float a = fabsf(v.hi);
  const unsigned b = __float_as_uint(a);
  const float half = __uint_as_float(b & 0x7F800000u) * 5.9604644775390625e-8f;  // ulp / 2
  const float err = a * (9.094947e-13f + 3.5527137e-15f / fabsf(c.hi));
  *out = v.hi;
  return a > 1e-20f && (b & 0x007FFFFFu) != 0u && fabsf(v.lo) < half * 0.99999f - err;
}

}  // namespace
}  // namespace ecpic
