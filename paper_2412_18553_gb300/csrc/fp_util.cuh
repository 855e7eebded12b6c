// Small floating-point helpers shared by the kernels: conversions that keep off
// the float64 units, and packed FP32 arithmetic.
#pragma once
#include <cstdint>

namespace te {

// float64 conversions share GB300's two float64 lanes per SM with the arithmetic
// (64 issue cycles of a scheduler each); the usual range is converted by integer
// operations instead (same bits).  The rare conversions are volatile so that
// the compiler does not issue them ahead of their branch.
__device__ __forceinline__ double cvt_double(float f) {
  double d;
  asm volatile("cvt.f64.f32 %0, %1;" : "=d"(d) : "f"(f));
  return d;
}
__device__ __forceinline__ float cvt_float(double d) {
  float f;
  asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(f) : "d"(d));
  return f;
}
__device__ __forceinline__ double to_double(float f) {
  const uint32_t u = __float_as_uint(f), m = u & 0x7FFFFFFFu;
  if (m - 0x00800000u < 0x7F000000u)  // normal
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(m << 29));
  return cvt_double(f);
}

// 2^e (h + l) as a float64 for |l| < ulp(h), by integer operations (about 25
// against two float64 operations of 64 issue cycles each): l shifted to h's
// 53-bit grid, rounded to nearest (ties up), and added to h's mantissa; a
// difference below h's power of two goes to the grid of the next lower one.
// A zero pair (what decayed integrals leave) gives zero.  Where all that does not
// hold (values below 2^-71, results out of the normal
// range, a sum that may cross a power of two) *other is set and the result is void:
// pair_convert then, in a branch of several elements that the compiler does not
// turn into predicated float64 work.
__device__ __forceinline__ double pair_double(float h, float l, int e, bool* other) {
  const uint32_t uh = __float_as_uint(h), ul = __float_as_uint(l), m = uh & 0x7FFFFFu;
  const int eh = (int)((uh >> 23) & 255u), d = eh - (int)((ul >> 23) & 255u), ed = eh + 896 + e;
  const bool zero = ((uh | ul) << 1) == 0u;
  if (!zero && (eh < 56 || eh == 255 || d < 23 || (d == 23 && ((m + 1u) & 0x7FFFFFu) <= 2u) || (uint32_t)(ed - 2) >= 2040u))
    *other = true;
  const bool minus = ((uh ^ ul) >> 31) != 0u;
  const uint32_t t = (((ul & 0x7FFFFFu) | 0x800000u) << 8) >> min(max(d - 23, 0), 31);  // l in quarter units
  const uint32_t L = ((minus && m == 0u && d < 54 ? t : t >> 1) + 1u) >> 1;
  const unsigned long long b = (((unsigned long long)(((uint32_t)ed << 20) | (m >> 3))) << 32) | (m << 29);
  const unsigned long long r = (minus ? b - L : b + L) | ((unsigned long long)(uh & 0x80000000u) << 32);
  return zero ? 0.0 : __longlong_as_double((long long)r);
}
__device__ __forceinline__ double pair_convert(float h, float l, double scale) {
  double x;
  asm volatile("add.f64 %0, %1, %2;" : "=d"(x) : "d"(cvt_double(h)), "d"(cvt_double(l)));
  asm volatile("mul.f64 %0, %1, %2;" : "=d"(x) : "d"(x), "d"(scale));
  return x;
}

// FP32 reciprocal of D rounded to nearest, as a float64
__device__ __forceinline__ double recip_seed(double D) {
  const uint32_t h = (uint32_t)__double2hiint(D), m = h & 0x7FFFFFFFu;
  if (m - ((1023u - 100u) << 20) < (200u << 20)) {  // 2^-100 <= |D| < 2^100
    const unsigned long long b0 = ((unsigned long long)m << 32) | (uint32_t)__double2loint(D);
    const unsigned long long b = b0 + 0xFFFFFFFull + ((b0 >> 29) & 1ull);  // ties to even
    return to_double(__frcp_rn(__uint_as_float((h & 0x80000000u) | ((uint32_t)(b >> 29) - (896u << 23)))));
  }
  return cvt_double(__frcp_rn(cvt_float(D)));
}
// one Newton step towards 1 / D
__device__ __forceinline__ double recip_newton(double D, double r) { return fma(r, fma(-D, r, 1.0), r); }

// Two FP32 values in one 64-bit register (add.f32x2, fma.f32x2: both lanes
// rounded as the scalar instruction rounds, half the issue slots).
struct f2 {
  unsigned long long v;
};
__device__ __forceinline__ f2 f2_make(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2_get(f2 x, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(x.v));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
// a - b (one rounding: the product with -1 is exact)
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) { return f2_fma(b, f2{0xBF800000BF800000ull}, a); }
// s + e == a + b exactly in both lanes (Knuth)
__device__ __forceinline__ void f2_two_sum(f2 a, f2 b, f2& s, f2& e) {
  s = f2_add(a, b);
  const f2 bb = f2_sub(s, a);
  e = f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb));
}

}  // namespace te
