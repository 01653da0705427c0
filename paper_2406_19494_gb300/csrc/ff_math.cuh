// Two-float arithmetic ("ff": an unevaluated sum of two FP32 numbers, about 47 bits) for the small
// terms of the FP64 face fluxes, and its conversions from and to FP64 by integer operations.
//
// Why.  On this GPU a warp's FP64 instruction occupies the SM's FP64 pipe for 16 cycles, in which
// the SM's four schedulers issue 64 other instructions; an ff product or sum costs 7 to 11 FP32
// instructions and an FP64 <-> ff conversion about 12, so a term whose ff error is below the
// rounding of the FP64 sum it is added to costs several times less in ff.  Algorithms: Dekker's
// and Knuth's exact sums (Knuth, TAOCP vol. 2, 4.2.2; Dekker, Numer. Math. 18, 1971) with the
// fused multiply-add as the exact product's second part.  Every operation is a round-to-nearest
// intrinsic, so that no compiler contraction changes a result and all kernels give the same bits.
#pragma once

#include <cmath>
#include <cstring>

#include "fast_math.cuh"

namespace fl {

struct ff {
  float h, l;
};

#ifdef __CUDA_ARCH__
FL_HD float s_add(float a, float b) { return __fadd_rn(a, b); }
FL_HD float s_sub(float a, float b) { return __fsub_rn(a, b); }
FL_HD float s_mul(float a, float b) { return __fmul_rn(a, b); }
FL_HD float s_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
FL_HD float s_rcp(float a) { float r; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a)); return r; }
FL_HD float s_rsqrt(float a) { float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a)); return r; }
FL_HD int s_bits(float a) { return __float_as_int(a); }
FL_HD float s_from(int a) { return __int_as_float(a); }
FL_HD int d_hi(double a) { return __double2hiint(a); }
FL_HD int d_lo(double a) { return __double2loint(a); }
FL_HD double d_from(int hi, int lo) { return __hiloint2double(hi, lo); }
#else
// host forms (the host-compiled checks; build them without floating-point contraction)
FL_HD float s_add(float a, float b) { return a + b; }
FL_HD float s_sub(float a, float b) { return a - b; }
FL_HD float s_mul(float a, float b) { return a * b; }
FL_HD float s_fma(float a, float b, float c) { return fmaf(a, b, c); }
FL_HD float s_rcp(float a) { return 1.0f / a; }
FL_HD float s_rsqrt(float a) { return 1.0f / sqrtf(a); }
FL_HD int s_bits(float a) { int i; memcpy(&i, &a, 4); return i; }
FL_HD float s_from(int a) { float f; memcpy(&f, &a, 4); return f; }
FL_HD int d_hi(double a) { long long i; memcpy(&i, &a, 8); return (int)(i >> 32); }
FL_HD int d_lo(double a) { long long i; memcpy(&i, &a, 8); return (int)i; }
FL_HD double d_from(int hi, int lo) {
  const unsigned long long i = ((unsigned long long)(unsigned)hi << 32) | (unsigned)lo;
  double d; memcpy(&d, &i, 8); return d;
}
#endif

// s + e = a + b exactly
FL_HD ff two_sum(float a, float b) {
  const float s = s_add(a, b), bb = s_sub(s, a);
  return {s, s_add(s_sub(a, s_sub(s, bb)), s_sub(b, bb))};
}
// the same for |a| >= |b| (or a = 0)
FL_HD ff quick_sum(float a, float b) {
  const float s = s_add(a, b);
  return {s, s_sub(b, s_sub(s, a))};
}

// Operators give normalised pairs (|l| <= 2^-24 |h| about): sums with an absolute error about
// 2^-48 (|a| + |b|), products with a relative error about 2^-47.
FL_HD ff ff_norm(ff a) { return two_sum(a.h, a.l); }
// the value rounded to FP32; its sign is the pair's
FL_HD float ff_float(ff a) { return s_add(a.h, a.l); }
FL_HD ff operator-(ff a) { return {-a.h, -a.l}; }
FL_HD ff operator+(ff a, ff b) {
  const ff s = two_sum(a.h, b.h);
  return quick_sum(s.h, s_add(s.l, s_add(a.l, b.l)));
}
FL_HD ff operator-(ff a, ff b) { return a + (-b); }
FL_HD ff operator+(ff a, float b) {
  const ff s = two_sum(a.h, b);
  return quick_sum(s.h, s_add(s.l, a.l));
}
FL_HD ff operator*(ff a, ff b) {
  const float p = s_mul(a.h, b.h);
  return quick_sum(p, s_fma(a.l, b.h, s_fma(a.h, b.l, s_fma(a.h, b.h, -p))));
}
FL_HD ff ff_sqr(ff a) {
  const float p = s_mul(a.h, a.h);
  return quick_sum(p, s_fma(s_add(a.h, a.h), a.l, s_fma(a.h, a.h, -p)));
}
// times a power of two (exact)
FL_HD ff ff_scale(ff a, float p2) { return {s_mul(a.h, p2), s_mul(a.l, p2)}; }
FL_HD ff ff_twice(ff a) { return {s_add(a.h, a.h), s_add(a.l, a.l)}; }
// a * b + c
FL_HD ff ff_fma(ff a, ff b, ff c) {
  const float p = s_mul(a.h, b.h);
  const float e = s_fma(a.l, b.h, s_fma(a.h, b.l, s_fma(a.h, b.h, -p)));
  const ff s = two_sum(p, c.h);
  return quick_sum(s.h, s_add(s.l, s_add(e, c.l)));
}
// The same without the renormalisation, three instructions fewer: |l| is then a few 2^-24 |h| (a later
// product drops l l, 2^-46 of it) or, where the sum cancelled, a few 2^-24 of the operands.
FL_HD ff add_weak(ff a, ff b) {
  const ff s = two_sum(a.h, b.h);
  return {s.h, s_add(s.l, s_add(a.l, b.l))};
}
FL_HD ff mul_weak(ff a, ff b) {
  const float p = s_mul(a.h, b.h);
  return {p, s_fma(a.l, b.h, s_fma(a.h, b.l, s_fma(a.h, b.h, -p)))};
}
FL_HD ff mul_weak(ff a, float b) {
  const float p = s_mul(a.h, b);
  return {p, s_fma(a.l, b, s_fma(a.h, b, -p))};
}
FL_HD ff sqr_weak(ff a) {
  const float p = s_mul(a.h, a.h);
  return {p, s_fma(s_add(a.h, a.h), a.l, s_fma(a.h, a.h, -p))};
}
FL_HD ff fma_weak(ff a, ff b, ff c) {
  const float p = s_mul(a.h, b.h);
  const float e = s_fma(a.l, b.h, s_fma(a.h, b.l, s_fma(a.h, b.h, -p)));
  const ff s = two_sum(p, c.h);
  return {s.h, s_add(s.l, s_add(e, c.l))};
}
// 1 / a from the FP32 estimate r: with e = 1 - a r, 1/a = r (1 + e + e^2 + O(e^3)), |e| < 2^-21
FL_HD ff ff_rcp(ff a) {
  const float r = s_rcp(a.h);
  const float e = s_fma(-a.l, r, s_fma(-a.h, r, 1.0f));
  return {r, s_mul(r, s_fma(e, e, e))};
}
// n / d
FL_HD ff ff_div(ff n, ff d) { return n * ff_rcp(d); }
// sqrt(a), a > 0: s = a y from the FP32 estimate y of 1/sqrt(a), then s + (a - s^2) y / 2
FL_HD ff ff_sqrt(ff a) {
  const float y = s_rsqrt(a.h), s = s_mul(a.h, y);
  const float e = s_add(s_fma(-s, s, a.h), a.l);
  return quick_sum(s, s_mul(s_mul(0.5f, y), e));
}

// x = h + l (1 + 2^-48): the leading 24 bits exact, the other 29 rounded to FP32.  |x| < 2^-126
// gives 0 or a subnormal number; |x| >= 2^127 or a non-finite x a number near 2^127, which no limit of
// the ff path admits.  P: the same of x 2^P, at no more operations.
template <int P = 0>
FL_HD ff ff_of(double x) {
  const int hw = d_hi(x), lw = d_lo(x);
  int t = (hw & 0x7fffffff) - ((1023 - 127 - P) << 20);             // exponent rebiased to FP32
  t = t < 0 ? 0 : (t > 0x0fefffff ? 0x0fefffff : t);
  const int h = (hw & (int)0x80000000u) | (t << 3) | (int)((unsigned)lw >> 29);
  // the low 29 fraction bits in units of 2^-52 of h's binade
  const float m = s_mul((float)(lw & 0x1fffffff), 2.220446049250313e-16f);
  return {s_from(h), s_mul(m, s_from(h & (int)0xff800000u))};
}

// h + l as FP64 for a normalised pair, within 2^-52 of it: h's bits widened, then l added in units
// of the result's last place.  The bit pattern of a double grows by one per unit in the last
// place, so the addition is an integer one; below a power of two the unit is half as large.
// |h| < 2^-70 gives h rounded to a few bits or 0; an infinite h or a NaN gives NaN.
FL_HD double ff_to_double(ff a) {
  const int u = s_bits(a.h);
  const int e = u & 0x7f800000;
  // below 2^-70 the binade of 2^-70 stands in: the value is far below any use
  const int eb = e < (57 << 23) ? (57 << 23) : e;
  int hi = (u & (int)0x80000000u) | (((u & 0x7fffffff) >> 3) + (e == 0 ? 0 : (1023 - 127) << 20));
  if (e == 0x7f800000) hi = 0x7ff80000;
  const int lo = u << 29;
  float k = s_mul(a.l, s_from((306 << 23) - eb));               // l times 2^(52 - (e - 127))
  // same sign as h: away from zero
  if (u < 0) k = -k;
  if ((u & 0x7fffff) == 0 && k < 0.0f) k = s_add(k, k);
#ifdef __CUDA_ARCH__
  const int i = __float2int_rn(k);
#else
  const int i = (int)rintf(k);
#endif
  const long long bits = (((long long)hi << 32) | (unsigned)lo) + (long long)i;
  return d_from((int)(bits >> 32), (int)bits);
}

}  // namespace fl
