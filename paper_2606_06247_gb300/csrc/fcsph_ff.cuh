// Double-float ("FP32x2") arithmetic: a value is the unevaluated sum hi + lo of
// two FP32 numbers (|lo| <= ulp(hi)/2), a 48-bit significand carried by the
// FP32 units.  GB300 runs FP32 at 64x its FP64 rate, so transforms in this
// format reach FP64-class rounding (unit roundoff ~2^-48) at FP32-unit speed.
//
// Building blocks are the classical error-free transformations (Knuth's
// TwoSum, Dekker's Fast2Sum, the FMA-based exact product); every operation
// uses the _rn intrinsics, which the compiler never contracts or reorders.
#pragma once

#include <cuda_runtime.h>

namespace fcsph {

// Exact conversions between FP64 and FP32 on the integer units.  The
// conversion instructions and every FP64 operation share 2 lanes per SM (the
// column passes kept them 29 % busy, 12 of 22 of those operations being
// conversions); the integer forms take normal numbers in FP32 range and zeros,
// the instruction the rest.
__device__ __forceinline__ double f2d(float x) {
  const unsigned u = __float_as_uint(x), m = u & 0x7fffffffu;
  if (m - 0x00800000u < 0x7f000000u)  // normal
    return __hiloint2double((int)((u & 0x80000000u) | ((m >> 3) + 0x38000000u)), (int)(u << 29));
  if (m == 0) return __hiloint2double((int)u, 0);
  return (double)x;
}
// h = fl(d), l = fl(d - h)
__device__ __forceinline__ void d2ff(double d, float& h, float& l) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned e = (hi >> 20) & 0x7ffu;
  if (e - (1023u - 60u) < 180u) {  // 2^-60 <= |d| < 2^120: h and l are normal (or l is zero)
    const unsigned sign = hi & 0x80000000u;
    const unsigned f = __funnelshift_l(lo, hi, 3) & 0x7fffffffu;  // exponent and mantissa above the 29 low bits
    const unsigned low = lo & 0x1fffffffu;
    const unsigned up = (low + 0x0fffffffu + (f & 1u)) >> 29;      // round to nearest, ties to even
    h = __uint_as_float((f - 0x40000000u + up) & 0x7fffffffu | sign);
    // the remainder low - up 2^29 in units of 2^(e - 1075), rounded to FP32
    const float r = __int2float_rn((int)low - (int)(up << 29));
    l = r * __uint_as_float(((e - 1075u + 127u) << 23) | sign);
  } else if (((hi & 0x7fffffffu) | lo) == 0u) {
    h = __uint_as_float(hi);
    l = 0.f;
  } else {
    h = (float)d;
    l = (float)(d - (double)h);
  }
}

struct ff {
  float h, l;
  __host__ __device__ ff() : h(0.f), l(0.f) {}
  // plain conversions, so that constant arguments fold at compile time
  __host__ __device__ ff(double d) : h((float)d), l((float)(d - (double)(float)d)) {}
  // exact for |i| < 2^24 (wavenumber indices), without a trip through FP64
  __host__ __device__ ff(int i) : h((float)i), l(0.f) {}
  __device__ explicit operator double() const { return f2d(h) + f2d(l); }
  __host__ __device__ explicit operator float() const { return h + l; }
};

__device__ __forceinline__ ff ff_from(double d) {
  ff r;
  d2ff(d, r.h, r.l);
  return r;
}
__device__ __forceinline__ ff ff_make(float h, float l) {
  ff r;
  r.h = h;
  r.l = l;
  return r;
}

// s + e = a + b exactly (no assumption on |a| vs |b|)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// s + e = a + b exactly when |a| >= |b|
__device__ __forceinline__ void fast_two_sum(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

__device__ __forceinline__ ff operator+(ff a, ff b) {
  float s, e;
  two_sum(a.h, b.h, s, e);
  e = __fadd_rn(e, __fadd_rn(a.l, b.l));
  float h, l;
  fast_two_sum(s, e, h, l);
  return ff_make(h, l);
}

__device__ __forceinline__ ff operator-(ff a) { return ff_make(-a.h, -a.l); }

__device__ __forceinline__ ff operator-(ff a, ff b) { return a + (-b); }

__device__ __forceinline__ ff operator*(ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);  // exact low part of a.h * b.h
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  float h, l;
  fast_two_sum(p, e, h, l);
  return ff_make(h, l);
}

__device__ __forceinline__ ff& operator+=(ff& a, ff b) {
  a = a + b;
  return a;
}

// a / b: FP32 quotient, one correction from the double-float remainder.
__device__ __forceinline__ ff operator/(ff a, ff b) {
  const float q1 = __fdiv_rn(a.h, b.h);
  const ff r = a - b * ff_make(q1, 0.f);
  const float q2 = __fdiv_rn(r.h, b.h);
  float h, l;
  fast_two_sum(q1, q2, h, l);
  return ff_make(h, l);
}

// A complex FP32-pair value: both high words, then both low words, so that
// every step of the pair arithmetic runs on the two components at once with
// the packed FP32 instructions (add / mul / fma.rn.f32x2: two FP32 results per
// issued instruction, each rounded as the scalar instruction rounds it; the
// pipe still takes two cycles for them, measured 64 packed against 128 scalar
// adds per clock and SM).  The pair transforms were bound by what 12 warps an
// SM can issue, not by the FP32 pipe (33 % busy at 47 % of issue slots used).
struct alignas(16) ff2 {
  float2 h, l;
};
__device__ __forceinline__ ff cre(ff2 a) { return ff_make(a.h.x, a.l.x); }
__device__ __forceinline__ ff cim(ff2 a) { return ff_make(a.h.y, a.l.y); }
__device__ __forceinline__ ff2 ff2_make(ff x, ff y) {
  ff2 r;
  r.h = make_float2(x.h, y.h);
  r.l = make_float2(x.l, y.l);
  return r;
}

// Packed FP32 arithmetic, componentwise and round-to-nearest.
__device__ __forceinline__ unsigned long long f2bits(float2 a) {
  return ((unsigned long long)__float_as_uint(a.y) << 32) | __float_as_uint(a.x);
}
__device__ __forceinline__ float2 bits2f(unsigned long long a) {
  return make_float2(__uint_as_float((unsigned)a), __uint_as_float((unsigned)(a >> 32)));
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2bits(a)), "l"(f2bits(b)));
  return bits2f(d);
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2bits(a)), "l"(f2bits(b)));
  return bits2f(d);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2bits(a)), "l"(f2bits(b)));
  return bits2f(d);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2bits(a)), "l"(f2bits(b)), "l"(f2bits(c)));
  return bits2f(d);
}
// sign changes on the integer units (the FP32 pipe is the busy one)
__device__ __forceinline__ float fneg(float a) { return __uint_as_float(__float_as_uint(a) ^ 0x80000000u); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(fneg(a.x), fneg(a.y)); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }

// s + e = a + b exactly, componentwise (two_sum); s - e form for a - b.
__device__ __forceinline__ void two_sum2(float2 a, float2 b, float2& s, float2& e) {
  s = add2(a, b);
  const float2 bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
}
__device__ __forceinline__ void two_diff2(float2 a, float2 b, float2& s, float2& e) {
  s = sub2(a, b);
  const float2 bb = sub2(s, a);
  e = sub2(sub2(a, sub2(s, bb)), add2(b, bb));
}
__device__ __forceinline__ ff2 norm2(float2 s, float2 e) {  // Fast2Sum, |s| >= |e|
  ff2 r;
  r.h = add2(s, e);
  r.l = sub2(e, sub2(r.h, s));
  return r;
}

// Butterfly-internal complex sums without the closing renormalisation: high
// words fl(a.h + b.h), low words their exact error plus a.l + b.l, so |low| may
// exceed ulp(high)/2 by a few ulps; and the renormalisation applied when a
// butterfly's outputs are stored.
__device__ __forceinline__ ff2 cadd_nr(ff2 a, ff2 b) {
  ff2 r;
  float2 e;
  two_sum2(a.h, b.h, r.h, e);
  r.l = add2(e, add2(a.l, b.l));
  return r;
}
__device__ __forceinline__ ff2 csub_nr(ff2 a, ff2 b) {
  ff2 r;
  float2 e;
  two_diff2(a.h, b.h, r.h, e);
  r.l = add2(e, sub2(a.l, b.l));
  return r;
}
__device__ __forceinline__ ff2 cnorm(ff2 a) { return norm2(a.h, a.l); }
__device__ __forceinline__ ff2 cadd(ff2 a, ff2 b) { return cnorm(cadd_nr(a, b)); }
__device__ __forceinline__ ff2 csub(ff2 a, ff2 b) { return cnorm(csub_nr(a, b)); }
__device__ __forceinline__ ff2 cconj(ff2 a) {
  a.h.y = fneg(a.h.y);
  a.l.y = fneg(a.l.y);
  return a;
}
// -i a, i a
__device__ __forceinline__ ff2 crot_m(ff2 a) {
  ff2 r;
  r.h = make_float2(a.h.y, fneg(a.h.x));
  r.l = make_float2(a.l.y, fneg(a.l.x));
  return r;
}
__device__ __forceinline__ ff2 crot_p(ff2 a) {
  ff2 r;
  r.h = make_float2(fneg(a.h.y), a.h.x);
  r.l = make_float2(fneg(a.l.y), a.l.x);
  return r;
}

// Exact product of the high words (p + its error) plus the cross terms:
// p + e ~ a * c componentwise, e = fma(a.h, c.h, -p) + a.h c.l + a.l c.h in
// the order of operator*.
__device__ __forceinline__ void prod2(ff2 a, float2 ch, float2 cl, float2& p, float2& e) {
  p = mul2(a.h, ch);
  e = fma2(a.h, ch, neg2(p));
  e = fma2(a.h, cl, e);
  e = fma2(a.l, ch, e);
}
// a * b + c * d with both exact products' high words through one TwoSum and
// the error terms added once, unrenormalised, for both components of a complex
// product: (a.x, a.y) b.x + (-a.y, a.x) b.y.
__device__ __forceinline__ ff2 cmul_nr(ff2 a, ff2 b) {
  float2 p1, e1, p2, e2, t;
  prod2(a, dup2(b.h.x), dup2(b.l.x), p1, e1);
  prod2(crot_p(a), dup2(b.h.y), dup2(b.l.y), p2, e2);
  ff2 r;
  two_sum2(p1, p2, r.h, t);
  r.l = add2(t, add2(e1, e2));
  return r;
}
__device__ __forceinline__ ff2 cmul(ff2 a, ff2 b) { return cnorm(cmul_nr(a, b)); }
__device__ __forceinline__ ff2 cmulc(ff2 a, ff2 b) { return cmul(a, cconj(b)); }  // a * conj(b)
// a * s (data times a real factor; the factor first in cscale_l, as in s * a:
// the cross terms are added in the other order)
__device__ __forceinline__ ff2 cscale(ff2 a, ff s) {
  float2 p, e;
  prod2(a, dup2(s.h), dup2(s.l), p, e);
  return norm2(p, e);
}
__device__ __forceinline__ ff2 cscale_l(ff s, ff2 a) {
  const float2 sh = dup2(s.h), sl = dup2(s.l);
  const float2 p = mul2(sh, a.h);
  float2 e = fma2(sh, a.h, neg2(p));
  e = fma2(sh, a.l, e);
  e = fma2(sl, a.h, e);
  return norm2(p, e);
}
// a / 2 (exact: the renormalised product of operator* gives the same pair)
__device__ __forceinline__ ff2 chalf(ff2 a) {
  a.h = mul2(a.h, dup2(0.5f));
  a.l = mul2(a.l, dup2(0.5f));
  return a;
}
// acc + a * c and a * c for a real constant c, unrenormalised (on
// both components; without an accumulator the sum with zero is exact).
__device__ __forceinline__ ff2 cmadd_nr(ff2 acc, ff2 a, ff c) {
  float2 p, e, t;
  prod2(a, dup2(c.h), dup2(c.l), p, e);
  ff2 r;
  two_sum2(acc.h, p, r.h, t);
  r.l = add2(t, add2(acc.l, e));
  return r;
}
__device__ __forceinline__ ff2 cmul0_nr(ff2 a, ff c) {
  ff2 r;
  prod2(a, dup2(c.h), dup2(c.l), r.h, r.l);
  return r;
}

}  // namespace fcsph
