// pf_ff.cuh -- pairs of floats ("ff": an unevaluated sum h + l, |l| <= ulp(h)/2)
// on the FP32 pipe.  GB300 issues 128 FP32 lanes a clock per SM and two FP64
// lanes, so one FP64 instruction costs the time of 64 FP32 ones; an ff
// product takes 7 and an ff sum 11, at 2^-47 relative instead of 2^-53.  The
// propagation kernels do in ff what is corrected later or is small beside the
// state it is added to, and keep the states and the last residual in FP64
// (pf_fast.cuh says where the line lies and why the result is as accurate).
//
// The error-free sums are Knuth's (TAOCP 4.2.2) and Dekker's (1971), the
// products' errors come from a fused multiply-add.  The operations must be
// rounded one by one, so they are written with the rounding intrinsics, which
// the compiler does not contract.  Conversions between double and ff are done
// on the integer pipe: the conversion instructions between the two formats run
// at the FP64 rate (two lanes a clock, measured).
//
// A host build (tests) gives the same bits but for the reciprocal's last one and the sign
// of a NaN.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define PF_FF_FN __device__ __forceinline__
#else
#include <cmath>
#define PF_FF_FN inline
#endif

namespace pfg {

struct ff {
  float h, l;
};

#ifdef __CUDACC__
PF_FF_FN float f_add(float a, float b) { return __fadd_rn(a, b); }
PF_FF_FN float f_sub(float a, float b) { return __fsub_rn(a, b); }
PF_FF_FN float f_mul(float a, float b) { return __fmul_rn(a, b); }
PF_FF_FN float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
PF_FF_FN uint32_t f_bits(float a) { return __float_as_uint(a); }
PF_FF_FN float f_from_bits(uint32_t b) { return __uint_as_float(b); }
PF_FF_FN uint32_t d_hi(double a) { return (uint32_t)__double2hiint(a); }
PF_FF_FN uint32_t d_lo(double a) { return (uint32_t)__double2loint(a); }
PF_FF_FN double d_from(uint32_t hi, uint32_t lo) { return __hiloint2double((int)hi, (int)lo); }
PF_FF_FN uint32_t shift_in(uint32_t hi, uint32_t lo, int s) { return __funnelshift_l(lo, hi, s); }
// hardware reciprocal, one ulp or so
PF_FF_FN float f_rcp(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}
#else
inline float f_add(float a, float b) { return a + b; }
inline float f_sub(float a, float b) { return a - b; }
inline float f_mul(float a, float b) { return a * b; }
inline float f_fma(float a, float b, float c) { return std::fma(a, b, c); }
inline uint32_t f_bits(float a) { uint32_t b; std::memcpy(&b, &a, 4); return b; }
inline float f_from_bits(uint32_t b) { float a; std::memcpy(&a, &b, 4); return a; }
inline uint32_t d_hi(double a) { uint64_t b; std::memcpy(&b, &a, 8); return (uint32_t)(b >> 32); }
inline uint32_t d_lo(double a) { uint64_t b; std::memcpy(&b, &a, 8); return (uint32_t)b; }
inline double d_from(uint32_t hi, uint32_t lo) {
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double a;
  std::memcpy(&a, &b, 8);
  return a;
}
inline uint32_t shift_in(uint32_t hi, uint32_t lo, int s) { return (hi << s) | (lo >> (32 - s)); }
inline float f_rcp(float a) { return 1.0f / a; }
#endif

// ------------------------------------------------------------------- sums
// s + e = a + b exactly
PF_FF_FN ff two_sum(float a, float b) {
  const float s = f_add(a, b), bb = f_sub(s, a);
  return ff{s, f_add(f_sub(a, f_sub(s, bb)), f_sub(b, bb))};
}
// the same for |a| >= |b| (or a = 0)
PF_FF_FN ff fast_two_sum(float a, float b) {
  const float s = f_add(a, b);
  return ff{s, f_sub(b, f_sub(s, a))};
}

PF_FF_FN ff ff_neg(ff a) { return ff{-a.h, -a.l}; }
PF_FF_FN ff ff_twice(ff a) { return ff{f_add(a.h, a.h), f_add(a.l, a.l)}; }

PF_FF_FN ff ff_add(ff a, ff b) {
  const ff s = two_sum(a.h, b.h);
  return fast_two_sum(s.h, f_add(s.l, f_add(a.l, b.l)));
}
PF_FF_FN ff ff_sub(ff a, ff b) { return ff_add(a, ff_neg(b)); }
PF_FF_FN ff ff_add(ff a, float b) {
  const ff s = two_sum(a.h, b);
  return fast_two_sum(s.h, f_add(s.l, a.l));
}
// a + b not renormalised (l up to h's size where they cancel), to 2^-45 of the larger
PF_FF_FN ff ff_add_raw(ff a, ff b) {
  const ff s = two_sum(a.h, b.h);
  return ff{s.h, f_add(s.l, f_add(a.l, b.l))};
}
PF_FF_FN ff ff_sub_raw(ff a, ff b) { return ff_add_raw(a, ff_neg(b)); }
// 1 + a
PF_FF_FN ff ff_one_plus(ff a) { return ff_add(a, 1.0f); }

// --------------------------------------------------------------- products
// a b, not renormalised (|l| a few ulps of h): for a sum that follows
PF_FF_FN ff ff_mul_raw(ff a, ff b) {
  const float p = f_mul(a.h, b.h);
  return ff{p, f_fma(a.h, b.l, f_fma(a.l, b.h, f_fma(a.h, b.h, -p)))};
}
PF_FF_FN ff ff_mul(ff a, ff b) {
  const ff p = ff_mul_raw(a, b);
  return fast_two_sum(p.h, p.l);
}
PF_FF_FN ff ff_mul(ff a, float b) {
  const float p = f_mul(a.h, b);
  return fast_two_sum(p, f_fma(a.l, b, f_fma(a.h, b, -p)));
}
// a b + c
PF_FF_FN ff ff_fma(ff a, ff b, ff c) { return ff_add(ff_mul_raw(a, b), c); }

// 1 / a: the hardware reciprocal and one Newton step on the pair
PF_FF_FN ff ff_rcp(ff a) {
  const float r = f_rcp(a.h);
  const float e = f_fma(-a.l, r, f_fma(-a.h, r, 1.0f));  // 1 - a r, exact product
  // r + r e + r e^2: |e| ~ 2^-23, so the last term is 2^-46 relative
  return fast_two_sum(r, f_mul(r, f_fma(e, e, e)));
}
// a / b: the quotient of the leading parts and its remainder's
PF_FF_FN ff ff_div(ff a, ff b) {
  const float r = f_rcp(b.h);
  const float q = f_mul(a.h, r);
  // a - q b: the leading product is exact in (p, e)
  const float p = f_mul(q, b.h), e = f_fma(q, b.h, -p);
  const float rem = f_add(f_sub(a.h, p), f_fma(-q, b.l, f_sub(a.l, e)));
  // the remainder is known to 2^-24 of itself times 2^-23 of a; its quotient
  // needs the reciprocal of all of b only to first order
  return fast_two_sum(q, f_mul(rem, r));
}

// ------------------------------------------------------------ conversions
// The pair nearest a double to about 2^-48 (h truncated).  |a| below 2^-126
// gives 0, |a| of 2^128 or more (or not finite) an infinite h.
PF_FF_FN ff ff_from(double a) {
  const uint32_t hi = d_hi(a), lo = d_lo(a);
  const uint32_t v = (hi & 0x7fffffffu) - 0x38000000u;
  uint32_t b = shift_in(v, lo, 3);
  // in range: 0x00100000 <= v < 0x0ff00000
  if (v - 0x00100000u >= 0x0fe00000u) b = (int32_t)v < 0x00100000 ? 0u : 0x7f800000u;
  b |= hi & 0x80000000u;
  // the 29 bits below h's, at the scale of h's exponent
  const float s = f_mul(f_from_bits(b & 0xff800000u), 0x1.0p-52f);
  return ff{f_from_bits(b), f_mul((float)(int32_t)(lo & 0x1fffffffu), s)};
}
// its leading float alone (truncated)
PF_FF_FN float f_from(double a) {
  const uint32_t hi = d_hi(a);
  const uint32_t v = (hi & 0x7fffffffu) - 0x38000000u;
  uint32_t b = shift_in(v, d_lo(a), 3);
  if (v - 0x00100000u >= 0x0fe00000u) b = (int32_t)v < 0x00100000 ? 0u : 0x7f800000u;
  return f_from_bits(b | (hi & 0x80000000u));
}
// exact for finite f; below the least normal float it gives 0 (an infinity or a NaN
// would become a number of 2^128: no caller passes one on)
PF_FF_FN double d_from_f(float f) {
  const uint32_t b = f_bits(f), m = b & 0x7fffffffu;
  const bool none = m < 0x00800000u;
  const uint32_t hi = none ? 0u : (m >> 3) + 0x38000000u;
  return d_from(hi | (b & 0x80000000u), none ? 0u : b << 29);
}

}  // namespace pfg
