// pf_math.cuh -- the logarithm and the sine/cosine pair of the Box-Muller
// transform in fewer FP64 instructions than the general-purpose library
// routines (on this chip every FP64 instruction counts): each is one table
// value and a short Taylor polynomial.
//
//  log x, after Tang (Table-driven implementation of the logarithm function
//  in IEEE floating-point arithmetic, ACM TOMS 16(4), 1990): x = 2^e y with
//  y in [1, 2), F = 1 + j/128 the breakpoint nearest y, f = y - F (exact),
//  r = f / F (as f times the tabulated 1/F), |r| <= 2^-8, and
//      log x = e log 2 + log F + log1p(r),
//  log1p(r) = r - r^2/2 + ... + r^7/7 (the next term is below 2^-67).  For x
//  in [1/2, 1) the first two terms are one tabulated value, log(F/2): as a sum
//  of two rounded constants it would cancel as F nears 2 (x just below 1).
//
//  sin(pi x), cos(pi x) for x = k 2^-52, 0 <= k < 2^53: the Box-Muller angle
//  2 pi u of a 53-bit uniform u = k 2^-53.  The nearest multiple j/64 of x is
//  split off exactly in integer arithmetic, x = j/64 + t with |t| <= 2^-7,
//  r = pi t, and the angle-addition formulas combine the tabulated sin, cos
//  of pi j/64 with sin r = r - r^3/3! + r^5/5! - r^7/7! and
//  cos r = 1 - r^2/2! + r^4/4! - r^6/6! (|r| <= pi/128; the next terms are
//  below 2^-66 and 2^-58).
//
// Both use only additions, multiplications and fused multiply-adds, so a host
// build of this header (plain C++) gives the same bits as the device one.
//
//  exp x and sqrt x without a single FP64 instruction (CUDA's take about 16 and 9
//  of them, the time of 1000 and 600 FP32 or integer ones; these take about 100
//  and 50), in fixed point with the small corrections in pairs of floats:
//  exp x, after Tang (Table-driven implementation of the exponential function in
//  IEEE floating-point arithmetic, ACM TOMS 15(2), 1989): x = n log 2/128 + r in
//  64-bit fixed point, exp x = 2^(n/128) (1 + p(r)), the table value of scale 2^61
//  times the polynomial in one 64x64-bit product, rounded once to a double.
//  sqrt x: the hardware's float approximation y of sqrt m, m in [1, 4), and two
//  Newton corrections m - y^2 over 2 y, the remainders exact in integers; the
//  sum, of unit 2^-52, is the result's mantissa.
//  With both in place (GB300): the scan of 2^20 weights 63 -> 32 us, the moments 89 ->
//  64 us, Robertson's stage 2 (N = 131072) 0.404 -> 0.373 ms, M1's (N = 50000) 0.144
//  -> 0.129 ms.
//  exp's host build gives the device's bits; sqrt's may differ from it in the last one
//  where the exact value is within 2^-16 ulp of a midpoint.
#pragma once
#include <stdint.h>

#include <math.h>
#include <string.h>

#include "pf_ff.cuh"
#include "pf_mathtab.h"

#ifdef __CUDACC__
#define PF_MATH_FN __device__ __forceinline__
#else
#define PF_MATH_FN inline
#endif

namespace pfm {

PF_MATH_FN int64_t bits_of(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  int64_t b;
  memcpy(&b, &x, sizeof b);
  return b;
#endif
}

PF_MATH_FN double from_bits(int64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  memcpy(&x, &b, sizeof x);
  return x;
#endif
}

// log x for a positive normal double x
PF_MATH_FN double log_pos(double x) {
  const int64_t b = bits_of(x);
  const int e = (int)(b >> 52) - 1023;
  const int64_t m = b & 0x000fffffffffffffLL;
  const int j = (int)((m + (1LL << 44)) >> 45);  // y's nearest j/128, 0..128
  const double y = from_bits(m | 0x3ff0000000000000LL);
  const double F = from_bits(0x3ff0000000000000LL + ((int64_t)j << 45));  // 1 + j/128
  const double r = (y - F) * kPfLogInvF[j];
  const double r2 = r * r;
  double p = fma(1.0 / 7.0, r, -1.0 / 6.0);
  p = fma(p, r, 1.0 / 5.0);
  p = fma(p, r, -1.0 / 4.0);
  p = fma(p, r, 1.0 / 3.0);
  p = fma(p, r, -0.5);
  const double l1p = fma(p, r2, r);
  const bool half = e == -1;
  return fma(half ? 0.0 : (double)e, 0x1.62e42fefa39efp-1, kPfLogF[j + (half ? 129 : 0)]) + l1p;
}

// The high 64 bits of a signed 64x64-bit product.
PF_MATH_FN int64_t mul_hi(int64_t a, int64_t b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (int64_t)(((__int128)a * b) >> 64);
#endif
}
PF_MATH_FN int32_t round_int(float v) {
#ifdef __CUDA_ARCH__
  return __float2int_rn(v);
#else
  return (int32_t)nearbyintf(v);
#endif
}
PF_MATH_FN float rsqrt_approx(float v) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
#else
  return 1.0f / sqrtf(v);
#endif
}

// (the rare cases, out of line)
#ifdef __CUDACC__
static __device__ __noinline__ double exp_edge(double x) { return exp(x); }
static __device__ __noinline__ double sqrt_edge(double x) { return sqrt(x); }
#else
inline double exp_edge(double x) { return exp(x); }
inline double sqrt_edge(double x) { return sqrt(x); }
#endif

// exp x, any x, within 0.6 ulp (results below 2^-1021 and values that are not
// finite: CUDA's exp).
PF_MATH_FN double exp_fixed(double x) {
  using namespace pfg;
  const uint32_t hi = d_hi(x), top = hi & 0x7fffffffu;
  // exp(-746) is below half the least denormal
  if (hi > 0xc0875000u && hi < 0xfff00000u) return 0.0;
  if (top >= 0x40860000u) return exp_edge(x);  // |x| >= 704, infinities, NaN
  // X = x 2^57 and n log 2/128 at that scale, modulo 2^64 (|x| reaches 2^9.5): their
  // difference is small
  const int sh = (int)(top >> 20) - 1018;  // of the 53-bit mantissa, at most 14
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | d_lo(x);
  const int rs = sh < -62 ? 62 : -sh;
  const uint64_t a = sh >= 0 ? m << sh : (m + ((1ull << rs) >> 1)) >> rs;
  const int n = round_int(f_mul(f_from(x), 0x1.715476p+7f));  // x 128/log 2
  const uint64_t X = (int32_t)hi < 0 ? 0ull - a : a;
  const int64_t low = ((int64_t)n * 3870238607LL + (1LL << 31)) >> 32;
  const int64_t R = (int64_t)(X - (uint64_t)(int64_t)n * 780414346020669ULL) - low;
  // p(r) = r + (r^2/2 + r^3/6 + r^4/24 + r^5/120), |r| <= 0.0028: the sum in pairs of
  // floats (r^2/2 <= 2^-18, wanted to 2^-60)
  const int32_t rh = (int32_t)(R >> 25);
  const ff r = fast_two_sum(f_mul((float)rh, 0x1p-32f), f_mul((float)(int32_t)(R - ((int64_t)rh << 25)), 0x1p-57f));
  const ff r2 = ff_mul(r, r);
  const float t = f_mul(f_mul(r.h, r.h), f_fma(r.h, 1.0f / 120.0f, 1.0f / 24.0f));
  const ff w = ff_add(ff_mul(r, ff{0x1.555556p-3f, -0x1.555556p-28f}), t);  // 1/6
  const ff q = ff_fma(r2, w, ff{0.5f * r2.h, 0.5f * r2.l});
  const int32_t q1 = round_int(f_mul(q.h, 0x1p42f));
  const float q2 = f_add(f_fma(q.h, 0x1p42f, -(float)q1), f_mul(q.l, 0x1p42f));
  const int64_t p62 = (R << 5) + ((int64_t)q1 << 20) + round_int(f_mul(q2, 0x1p20f));
  const int64_t T = kPfExp2[n & 127];
  const int64_t V = T + mul_hi(T, p62 << 2);  // of scale 2^61, in [2^61 (1 - 2^-8), 2^62 (1 + 2^-8))
  const int up = V >= (1LL << 62) ? 1 : V >= (1LL << 61) ? 0 : -1;
  const int64_t mant = (V + (1LL << (8 + up))) >> (9 + up);
  return from_bits(((int64_t)((n >> 7) + up + 1022) << 52) + mant);
}

// sqrt x within 0.501 ulp (zeros, denormals, negative values and values that are
// not finite: CUDA's sqrt).
PF_MATH_FN double sqrt_fixed(double x) {
  using namespace pfg;
  const uint32_t hi = d_hi(x);
  if (hi - 0x00100000u >= 0x7fe00000u) return sqrt_edge(x);
  const int odd = (int)(~hi >> 20) & 1;  // of the exponent without its bias
  const int64_t M = (int64_t)((((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | d_lo(x)) << odd);  // m 2^52
  const float mf = f_mul((float)(int32_t)(M >> 24), 0x1p-28f);
  const float r0 = rsqrt_approx(mf), h0 = f_mul(0.5f, r0);
  const float y = fminf(fmaxf(f_mul(mf, r0), 1.0f), 0x1.fffffep+0f);
  const int32_t Y = round_int(f_mul(y, 0x1p23f));  // exact
  const int64_t rem = M - (((int64_t)Y * Y) << 6);  // (m - y^2) 2^52
  // c = rem/(2 y): first to 2^-48, then the remainder of that
  const int32_t c1 = round_int(f_mul((float)(int32_t)(rem >> 4), h0));
  const int64_t rem2 = (rem << 18) - (int64_t)Y * c1 - (((int64_t)c1 * c1) >> 26);  // at 2^-70
  const int32_t c2 = round_int(f_mul(f_mul((float)(int32_t)rem2, h0), 0x1p-18f));
  const int64_t m52 = ((int64_t)Y << 29) + ((int64_t)c1 << 4) + c2;  // sqrt m 2^52, in [2^52, 2^53]
  const int he = ((int)(hi >> 20) - 1023 - odd) / 2;
  return from_bits(((int64_t)(he + 1022) << 52) + m52);
}

// sin(pi x) and cos(pi x), x = k 2^-52, k < 2^53
PF_MATH_FN void sincospi_k52(uint64_t k, double& s, double& c) {
  const int64_t j = (int64_t)((k + (1ULL << 45)) >> 46);  // x's nearest j/64, 0..128
  const int64_t rem = (int64_t)k - (j << 46);               // |rem| <= 2^45: exact as a double
  // r = pi rem 2^-52, with pi 2^-52 the double nearest pi times 2^-52
  const double r = (double)rem * 0x1.921fb54442d18p-51;
  const double r2 = r * r;
  double q = fma(r2, -1.0 / 5040.0, 1.0 / 120.0);
  q = fma(q, r2, -1.0 / 6.0);
  const double sr = fma(q, r2 * r, r);
  double u = fma(r2, -1.0 / 720.0, 1.0 / 24.0);
  u = fma(u, r2, -0.5);
  const double cr = fma(u, r2, 1.0);
  const double sa = kPfSinPi64[j], ca = kPfCosPi64[j];
  s = fma(sa, cr, ca * sr);
  c = fma(ca, cr, -(sa * sr));
}

}  // namespace pfm
