// Scalar building blocks that keep work off GB300's FP64 pipe.
//
// An SM has two FP64 lanes against 128 for FP32 and 64 or more for integers:
// one FP64 instruction of a warp occupies its pipe for 16 clocks, in which
// the SM's schedulers could issue 64 others.  What needs no 64-bit rounding
// (comparisons, selections, conversions between the float types, a Newton
// correction that is already small) therefore runs on the bits or in float;
// compares and conversions of doubles would take an FP64 slot each.
#pragma once
#include <cuda_runtime.h>

namespace rossbi {

// ---------------------------------------------------------------- doubles by their bits
__device__ __forceinline__ bool sign_bit(double x) { return __double2hiint(x) < 0; }
__device__ __forceinline__ bool sign_bit(float x) { return __float_as_int(x) < 0; }

// x > 0, false for NaN (the bits of +inf and below, above +0).
__device__ __forceinline__ bool positive(double x) {
  return (unsigned long long)(__double_as_longlong(x) - 1) < 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool positive(float x) { return x > 0.0f; }

// x >= 0, false for NaN.
__device__ __forceinline__ bool non_negative(double x) {
  return positive(x) || ((unsigned long long)__double_as_longlong(x) << 1) == 0;
}
__device__ __forceinline__ bool non_negative(float x) { return x >= 0.0f; }

// x is a positive normal number (not subnormal, infinite or NaN).
__device__ __forceinline__ bool positive_normal(double x) { return (unsigned)((__double2hiint(x) >> 20) - 1) < 0x7feu; }

// A dust cell has mass where its density is a normal number (or infinite): the
// reciprocal of a subnormal one may overflow.
__device__ __forceinline__ bool has_mass(double rho) {
  return (unsigned long long)(__double_as_longlong(rho) - 0x0010000000000000ll) <= 0x7fe0000000000000ull;
}
__device__ __forceinline__ bool has_mass(float rho) { return rho >= 0x1p-126f; }
// A dust density after a stage, negative subnormal ones as zero: a cell that has
// mass in the first stage's input but not in the second's leaves its neighbours
// short by less than the smallest normal number.
__device__ __forceinline__ double dust_density(double rho) {
  return (unsigned)__double2hiint(rho) >> 20 == 0x800u ? 0.0 : rho;
}
__device__ __forceinline__ float dust_density(float rho) { return rho > -0x1p-126f ? fmaxf(rho, 0.0f) : rho; }

// |a| < |b| (magnitudes of non-NaN values order like their bits).
__device__ __forceinline__ bool mag_less(double a, double b) {
  return (__double_as_longlong(a) & 0x7fffffffffffffffll) < (__double_as_longlong(b) & 0x7fffffffffffffffll);
}

// max(x, 0) and min(x, 0)
__device__ __forceinline__ double pos_part(double x) { return sign_bit(x) ? 0.0 : x; }
__device__ __forceinline__ double neg_part(double x) { return sign_bit(x) ? x : 0.0; }
__device__ __forceinline__ float pos_part(float x) { return fmaxf(x, 0.0f); }
__device__ __forceinline__ float neg_part(float x) { return fminf(x, 0.0f); }

// The smaller of two values of one sign in magnitude.
__device__ __forceinline__ double min_mag(double a, double b) { return mag_less(a, b) ? a : b; }

// x / 2^K for normal results, by the exponent (0 below the normal range).
template <int K>
__device__ __forceinline__ double scale_down(double x) {
  const int hi = __double2hiint(x);
  const bool normal = (hi & 0x7ff00000) > (K << 20);
  return __hiloint2double(normal ? hi - (K << 20) : (hi & 0x80000000), normal ? __double2loint(x) : 0);
}

// MinMod slope: 0 where the signs differ.
__device__ __forceinline__ double minmod_bits(double a, double b) {
  const double m = min_mag(a, b);
  return (__double2hiint(a) ^ __double2hiint(b)) < 0 ? 0.0 : m;
}

// min(|a|, |b|) with the sign of a * b (one instruction).
__device__ __forceinline__ float min_xorsign(float a, float b) {
  float r;
  asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// The smaller value, NaN if either is.
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// double -> float by truncation, flushed to 0 below and held at FLT_MAX above
// float's range; float -> double, exact for normal values, subnormals to 0.
// `bias` other than the formats' own 896 scales by a power of two on the way,
// narrow(x, 896 + k) = x / 2^k and widen(y, 896 + k) = y 2^k (0 < bias < 1792:
// zero stays zero, and the widened value is a normal number).
constexpr int FLOAT_BIAS = 896;
__device__ __forceinline__ int exponent(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ float narrow(double x, int bias = FLOAT_BIAS) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int e = exponent(x) - bias;
  unsigned b = __funnelshift_l(lo, hi & 0x7fffffffu, 3) - ((unsigned)bias << 23);
  b = (unsigned)(e - 1) < 254u ? b & 0x7fffffffu : (e < 1 ? 0u : 0x7f7fffffu);
  return __uint_as_float(b | (hi & 0x80000000u));
}
__device__ __forceinline__ float narrow(float x) { return x; }
__device__ __forceinline__ double widen(float x, int bias = FLOAT_BIAS) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned hi = m < 0x00800000u ? 0u : (m >> 3) + ((unsigned)bias << 20);
  return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(m < 0x00800000u ? 0u : b << 29));
}

// ---------------------------------------------------------------- reciprocals
// One step of the third-order Householder iteration (y (1 + e + e^2) with
// e = 1 - x y for 1/x; y (1 + e/2 + 3 e^2/8) with e = 1 - x y^2 for x^-1/2)
// from the PTX approximation, whose error of about 2^-20 it takes below
// 2^-59: three and five FP64 operations, where the correctly rounded division
// and square root with their scaling take 8 and more.  recip() takes every
// value: where the approximation is zero or not finite (zero, subnormal,
// infinite or NaN arguments and those above 2^1022) it divides.
__device__ __forceinline__ double recip(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  if ((unsigned)(exponent(y) - 1) >= 0x7feu) return 1.0 / x;
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
// x^-1/2 of a positive normal number.
__device__ __forceinline__ double recip_sqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}
// The hardware's approximation in float; recip_normal() without the scaling of
// subnormal arguments (infinite) and results (zero).
__device__ __forceinline__ float recip(float x) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float recip_normal(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float recip_sqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// One Newton step of 1/x and x^-1/2 from y (error e of y: e^2 and 3 e^2 / 2).
__device__ __forceinline__ double refine_recip(double x, double y) { return fma(y, fma(-x, y, 1.0), y); }
__device__ __forceinline__ double refine_recip_sqrt(double x, double y) {
  return fma(scale_down<1>(y), fma(-(x * y), y, 1.0), y);
}
// sqrt(x) of any x.  Squares of slow velocities underflow, so subnormal
// arguments are ordinary ones here, and the approximation flushes them to an
// infinite x^-1/2.
__device__ __forceinline__ double root(double x) {
  if (!positive_normal(x)) return sqrt(x);
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double t = x * y, e = fma(-t, y, 1.0);
  return fma(t * e, fma(0.375, e, 0.5), t);
}
__device__ __forceinline__ float root(float x) {
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return x >= 0x1p-126f && x <= 0x1.fffffep127f ? x * recip_sqrt(x) : y;
}

// ---------------------------------------------------------------- two floats at a time (the packed arithmetic of sm_100 and later)
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, pack2(-1.0f, -1.0f), a); }
}  // namespace rossbi
