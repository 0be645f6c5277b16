// FP64 functions of the splitting kinematics and the dipole cache, written
// for the cost of FP64 on this part: an FP64 instruction holds the SM's FP64
// pipe for 16 cycles whatever its active lanes, so what counts is their
// number.  The argument checks run on the bits, the seeds are single
// precision (MUFU) moved between the formats with integer instructions, and
// inputs outside a function's range take the CUDA library's function out of
// line, which also keeps these functions' code short: the kernels that call
// them are long enough to miss the instruction cache.
//
//   function          FP64 instructions   error
//   rcp_fp64          3                   0.51 ulp
//   div_fp64          6                   0.51 ulp
//   rsqrt_fp64        5                   0.51 ulp
//   sqrt_fp64         8                   0.51 ulp
//   exp_fp64          12                  0.55 ulp
//   expm1_neg_fp64    13                  1.6 ulp (near 2^(-1/64), where t - 1 and t p cancel in part)
//   circle_fp64       18                  1.2 ulp (sine and cosine; near the axes, from theta's own rounding)
// (bounds from the analyses below; the tests measure them on the device).
//
// Exponential: P. T. P. Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15
// (1989) 144-157, with 64 steps per octave, written from the method's
// description.  Sine and cosine: the angle addition theorem from the nearest
// of 64 tabulated points of the circle, with Taylor polynomials.  Reciprocal
// and reciprocal square root: a single-precision seed and one step of the
// geometric and binomial series, whose residual is exact or nearly so.
#pragma once

#include <cstdint>

#include "math_tables.inc"

namespace gaps {

struct alignas(16) ExpEntry {
  double hi, lo;
};
struct alignas(32) CircleEntry {
  double s, c, s_lo, c_lo;
};
static __device__ const ExpEntry kExpTable[] = {GAPS_EXP_TABLE};
static __device__ const CircleEntry kCircleTable[] = {GAPS_CIRCLE_TABLE};

static __device__ __noinline__ double exp_library(double x) { return exp(x); }
static __device__ __noinline__ double expm1_library(double x) { return expm1(x); }
static __device__ __noinline__ double rsqrt_library(double x) { return rsqrt(x); }
static __device__ __noinline__ double sqrt_library(double x) { return sqrt(x); }
static __device__ __noinline__ double div_library(double a, double d) { return a / d; }

// Positive x with an exponent within +-120, so that x, 1/x and their roots
// are normal single-precision numbers.
__device__ __forceinline__ bool seed_range(double x) {
  return static_cast<uint32_t>(__double2hiint(x)) - (903u << 20) < (240u << 20);
}
// x truncated to single precision (seed_range), and a normal positive
// single-precision number as a double (exact).
__device__ __forceinline__ float seed_of(double x) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)) - 0x38000000u;
  return __uint_as_float((hi << 3) | (static_cast<uint32_t>(__double2loint(x)) >> 29));
}
__device__ __forceinline__ double from_seed(float f) {
  const uint32_t b = __float_as_uint(f);
  return __hiloint2double(static_cast<int>((b >> 3) + 0x38000000u), static_cast<int>(b << 29));
}

// 1/d = r0 / (1 - e) = r0 (1 + e + e^2 + O(e^3)) with e = 1 - d r0, exact to
// the rounding of the fma; |e| < 2^-21, so e^3 < 2^-63.
__device__ __forceinline__ double rcp_seeded(double d) {
  const double r0 = from_seed(__fdividef(1.0f, seed_of(d)));
  const double e = fma(-d, r0, 1.0);
  return fma(r0, fma(e, e, e), r0);
}
__device__ __forceinline__ double rcp_fp64(double d) { return seed_range(d) ? rcp_seeded(d) : div_library(1.0, d); }
__device__ __forceinline__ double div_fp64(double a, double d) {
  if (!seed_range(d)) return div_library(a, d);
  const double r = rcp_seeded(d);
  const double q = a * r;
  return fma(fma(-d, q, a), r, q);
}

// x^-1/2 = y0 (1 - e)^-1/2 = y0 (1 + e/2 + 3 e^2/8 + O(e^3)) with
// e = 1 - x y0^2; y0 has 24 bits, so y0^2 is exact and e is exact to the
// rounding of the fma; |e| < 2^-20, so the rest is below 2^-61.
__device__ __forceinline__ double rsqrt_fp64(double x) {
  if (!seed_range(x)) return rsqrt_library(x);
  const double y0 = from_seed(rsqrtf(seed_of(x)));
  const double e = fma(-x, y0 * y0, 1.0);
  return fma(e * y0, fma(e, 0.375, 0.5), y0);
}
__device__ __forceinline__ double sqrt_fp64(double x) {
  if (!seed_range(x)) return sqrt_library(x);
  const double y0 = from_seed(rsqrtf(seed_of(x)));
  const double e = fma(-x, y0 * y0, 1.0);
  // x y0 in two parts: its own rounding would cost another half ulp
  const double h = x * y0, l = fma(x, y0, -h);
  return h + fma(e * h, fma(e, 0.375, 0.5), l);
}

// e^x = 2^m 2^(k/64) e^r with 64 m + k the integer nearest to 64 x / ln 2 and
// |r| <= ln 2 / 128: t + t_lo = 2^m 2^(k/64) and p = e^r - 1 by its Taylor
// polynomial to r^6 (the rest is below 2^-65, and below 2^-57 of p).
struct ExpParts {
  double t, t_lo, p;
};
__device__ __forceinline__ ExpParts exp_parts(double x) {
  constexpr double kMagic = 0x1.8p52;
  const double shifted = fma(x, GAPS_EXP_STEP_INV, kMagic);
  const int n = __double2loint(shifted);
  const double nd = shifted - kMagic;
  double r = fma(nd, -GAPS_EXP_STEP_HI, x);  // exact
  r = fma(nd, -GAPS_EXP_STEP_LO, r);
  const double2 e = __ldg(reinterpret_cast<const double2*>(&kExpTable[n & 63]));
  const int scale = (n >> 6) * (1 << 20);  // added to the exponent field
  ExpParts o;
  o.t = __hiloint2double(__double2hiint(e.x) + scale, __double2loint(e.x));
  // a zero remainder stays zero
  o.t_lo = __double2hiint(e.y) == 0 ? 0.0 : __hiloint2double(__double2hiint(e.y) + scale, __double2loint(e.y));
  double q = fma(r, 1.0 / 720.0, 1.0 / 120.0);
  q = fma(q, r, 1.0 / 24.0);
  q = fma(q, r, 1.0 / 6.0);
  q = fma(q, r, 0.5);
  o.p = fma(r * r, q, r);
  return o;
}
// |x| < 600 from its bits: t and its remainder stay normal numbers.
__device__ __forceinline__ bool exp_range(double x) {
  return (static_cast<uint32_t>(__double2hiint(x)) & 0x7fffffffu) < 0x4082c000u;
}
__device__ __forceinline__ double exp_fp64(double x) {
  if (!exp_range(x)) return exp_library(x);
  const ExpParts o = exp_parts(x);
  return o.t + fma(o.t, o.p, o.t_lo);
}
// e^x - 1 for x <= 0 (the t - 1 of t <= 1 is exact for t >= 1/2, and its
// rounding is within an ulp of the result below).
__device__ __forceinline__ double expm1_neg_fp64(double x) {
  if (!exp_range(x)) return expm1_library(x);
  const ExpParts o = exp_parts(x);
  return (o.t - 1.0) + fma(o.t, o.p, o.t_lo);
}
// Either of the two, chosen per lane, by the same instructions.
__device__ __forceinline__ double exp_or_expm1_fp64(double x, bool minus_one) {
  if (!exp_range(x)) return minus_one ? expm1_library(x) : exp_library(x);
  const ExpParts o = exp_parts(x);
  return (minus_one ? o.t - 1.0 : o.t) + fma(o.t, o.p, o.t_lo);
}

// Sine and cosine of 2 pi u for the 52-bit uniform u of (hi, lo), u itself
// given: the nearest k/64 comes from the top bits of hi, u - k/64 is exact,
// theta = 2 pi (u - k/64) <= pi/64 in magnitude; sin theta to theta^9 and
// cos theta - 1 to theta^8 (the rests below 2^-60 of them).
__device__ __forceinline__ void circle_fp64(double u, uint32_t hi, double* sn, double* cs) {
  const int k = static_cast<int>(((hi >> 25) + 1u) >> 1);
  const int top = 31 - __clz(k);  // k / 64 from its bits
  const int k64 = k == 0 ? 0 : ((1023 - 6 + top) << 20) | ((k << (20 - top)) & 0xfffff);
  const double d = u - __hiloint2double(k64, 0);
  const double th = GAPS_TWO_PI * d, t2 = th * th;
  double q = fma(t2, 1.0 / 362880.0, -1.0 / 5040.0);
  q = fma(q, t2, 1.0 / 120.0);
  q = fma(q, t2, -1.0 / 6.0);
  const double s = fma(th * t2, q, th);
  double c = fma(t2, 1.0 / 40320.0, -1.0 / 720.0);
  c = fma(c, t2, 1.0 / 24.0);
  c = fma(c, t2, -0.5);
  c = c * t2;  // cos theta - 1
  const double2* e = reinterpret_cast<const double2*>(&kCircleTable[k]);
  const double2 hi2 = __ldg(e), lo2 = __ldg(e + 1);
  *sn = hi2.x + fma(hi2.y, s, fma(hi2.x, c, lo2.x));
  *cs = hi2.y + fma(-hi2.x, s, fma(hi2.y, c, lo2.y));
}

}  // namespace gaps
