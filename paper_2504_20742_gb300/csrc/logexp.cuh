// logexp.cuh -- FP64 logarithm, exponential and square root for the phase-change source.
//
// The FP64 pipe bounds every kernel that evaluates the source (GB300 issues one FP64 warp
// instruction per SM every 16 cycles, 64 issue slots), so these spend integer and FP32
// instructions to save FP64 ones.  Table-driven argument reduction after Tang (ACM TOMS 16, 1990,
// "Table-driven implementation of the logarithm function"; TOMS 15, 1989, for the exponential):
// a 513-entry table leaves a reduced argument below 2^-10, whose third- and higher-order terms and
// the tables' low parts then fit FP32 arithmetic, and only the leading terms take FP64.
// FP64-pipe instructions per call (counted with ncu; CUDA's own in brackets): log_t 5 (29), exp_t
// 4 (15), expm1_t 7 (19), sqrt_t 5 (8), quot_t 4 (8).  Arguments outside the range of the fast
// form (zero, subnormal, negative, huge, infinite, NaN) take CUDA's function.
// Errors against 200-bit arithmetic: tests/test_gpu_logexp.py.
#pragma once
#include <cuda_runtime.h>
#include <math.h>

#include "fastmath.cuh"
#include "logexp_tables.cuh"

namespace ct {

// double -> float by truncation of the bits (normal results; smaller magnitudes give 0), and
// float -> double (exact for normal values; zero and subnormals give 0): the conversion
// instructions run on the FP64 pipe, these on the integer one.  For |x| < 2^127.
__device__ __forceinline__ float d2f_bits(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const unsigned a = h & 0x7fffffffu;
  const unsigned f = ((a - 0x38000000u) << 3) | (l >> 29);
  return __uint_as_float(a >= 0x38100000u ? (f | (h & 0x80000000u)) : 0u);
}
__device__ __forceinline__ double f2d_bits(float x) {
  const unsigned u = __float_as_uint(x), a = u & 0x7fffffffu;
  const unsigned h = (u & 0x80000000u) | ((a >> 3) + 0x38000000u);
  return __hiloint2double((int)(a >= 0x00800000u ? h : 0u), (int)(a >= 0x00800000u ? u << 29 : 0u));
}
// x / 2 on the integer pipe, for zero and normal x with a normal half: what the reductions below take
// (their r is zero or so large, or its square underflows whatever its half is)
__device__ __forceinline__ double half_normal(double x) {
  const int h = __double2hiint(x);
  return __hiloint2double(((unsigned)h & 0x7ff00000u) != 0u ? h - 0x00100000 : h, __double2loint(x));
}
// x / 2 on the integer pipe, for every x: one off the exponent; where that ends (zero, subnormals and
// the lowest normal binade share their scale), half of the bits, rounded to even.  Infinite and NaN
// values are returned as they are.
__device__ __forceinline__ double half_bits(double x) {
  const int h = __double2hiint(x);
  const unsigned e = (unsigned)h & 0x7ff00000u;
  if (e <= 0x00100000u) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x), m = b & 0x7fffffffffffffffull, q = m >> 1;
    return __longlong_as_double((long long)((b ^ m) | (q + (m & q & 1ull))));
  }
  return __hiloint2double(e != 0x7ff00000u ? h - 0x00100000 : h, __double2loint(x));
}

// CUDA's functions for the other arguments, out of line: their code (some 150 instructions each) is
// not repeated at every call
static __device__ __noinline__ double log_other(double x) { return log(x); }
static __device__ __noinline__ double exp_other(double x) { return exp(x); }
static __device__ __noinline__ double expm1_other(double x) { return expm1(x); }
static __device__ __noinline__ double sqrt_other(double x) { return sqrt(x); }
static __device__ __noinline__ double quot_other(double a, double b) { return a / b; }

// ln x.  x = 2^e m, k = round(1024 / m), r = m k/1024 - 1 (|r| <= 2^-10):
// ln x = e ln2 - ln(k/1024) + r - r^2/2 + [r^3/3 - r^4/4 + r^5/5 and the low parts, FP32].
__device__ __forceinline__ double log_t(double x) {
  const int hx = __double2hiint(x), lx = __double2loint(x);
  if ((unsigned)(hx - 0x00100000) >= 0x7fe00000u) return log_other(x);
  const double m = __hiloint2double((hx & 0x000fffff) | 0x3ff00000, lx);
  const float mf = __uint_as_float(0x3f800000u | (((unsigned)hx & 0x000fffffu) << 3) | ((unsigned)lx >> 29));
  const int k = __float2int_rn(__fdividef(1024.0f, mf)) - 512;
  const float ef = (float)((hx >> 20) - 1023);
  const double r = fma(m, __hiloint2double(0x3fe00000 + (k << 11), 0), -1.0);
  const float rf = d2f_bits(r);
  const float w = fmaf(rf * rf * rf, fmaf(rf, fmaf(rf, 0.2f, -0.25f), 0.33333334f), fmaf(ef, mtab::LN2_L, __ldg(mtab::LOG_LO + k)));
  const double s = fma(-half_normal(r), r, r);
  const double t = fma(f2d_bits(ef), mtab::LN2_H, __ldg(mtab::LOG_HI + k));   // exact
  return t + (s + f2d_bits(w));
}

// Reduction of the exponential: n = round(512 x / ln2), r = x - n ln2/512 (|r| <= 2^-10);
// e^x = 2^(n/512) (1 + s), s = r + r^2/2 + r^3/6 + [higher orders and the low parts, FP32].  CUBIC:
// the third-order term in FP64 too, for expm1, whose result is as small as r.  |x| < 700.
template <bool CUBIC>
__device__ __forceinline__ double exp_parts(double x, double& s) {
  const int n = __float2int_rn(d2f_bits(x) * 738.65986f);
  const float nf = (float)n;
  const int i = n & 511;
  const double r = fma(-f2d_bits(nf), mtab::L512_H, x);
  const float rf = d2f_bits(r), low = fmaf(-nf, mtab::L512_L, __ldg(mtab::EXP_LO + i));
  if (CUBIC) {
    const float w = fmaf(rf * rf * rf, fmaf(rf, 0.0083333338f, 0.041666668f) * rf, low);
    s = fma(r * r, fma(r, 1.0 / 6.0, 0.5), r) + f2d_bits(w);
  } else {
    const float w = fmaf(rf * rf * rf, fmaf(rf, 0.041666668f, 0.16666667f), low);
    s = fma(half_normal(r), r, r) + f2d_bits(w);
  }
  const double T = __ldg(mtab::EXP_HI + i);
  return __hiloint2double(__double2hiint(T) + ((n >> 9) << 20), __double2loint(T));
}
__device__ __forceinline__ bool exp_range(double x) { return (__double2hiint(x) & 0x7fffffff) < 0x4085e000; }   // |x| < 700
__device__ __forceinline__ double exp_t(double x) {
  if (!exp_range(x)) return x < -746.0 ? 0.0 : exp_other(x);   // most nucleation rates of a plume underflow
  double s;
  const double T = exp_parts<false>(x, s);
  return fma(T, s, T);
}
__device__ __forceinline__ double expm1_t(double x) {
  if (!exp_range(x)) return x < 0.0 ? -1.0 : expm1_other(x);
  double s;
  const double T = exp_parts<true>(x, s);
  return fma(T, s, T - 1.0);
}

// 1/b and a/b by one third-order Newton step from the hardware's approximate reciprocal (relative
// error below 2^-20, so its cube is below the rounding), for 2^-1000 <= |b| < 2^1000; IEEE
// division outside.
__device__ __forceinline__ bool rcp_range(double b) {
  return (((unsigned)__double2hiint(b) & 0x7ff00000u) - 0x01700000u) < 0x7d000000u;
}
__device__ __forceinline__ double rcp_t(double b) {
  if (!rcp_range(b)) return quot_other(1.0, b);
  double x;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(x) : "d"(b));
  const double e = fma(-b, x, 1.0);
  return fma(x, fma(e, e, e), x);
}
__device__ __forceinline__ double quot_t(double a, double b) {
  if (!rcp_range(b)) return quot_other(a, b);
  return a * rcp_t(b);
}

// sqrt x by one third-order step from the approximate reciprocal root, for 2^-1000 <= x < 2^1000
__device__ __forceinline__ double sqrt_t(double x) {
  if (!rcp_range(x) || __double2hiint(x) < 0) return sqrt_other(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y;
  const double e = fma(-t, y, 1.0);
  return fma(t * e, fma(0.375, e, 0.5), t);
}

}  // namespace ct
