// Device helpers: periodic index, principal-branch complex power for kappa(w) = 1 + c w^p, conversions between
// double and float.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

namespace frkc2 {

// A cell index on a periodic axis (g >= -n).
__device__ __forceinline__ int wrap3(int g, int n) {
  if (g < 0) g += n;
  while (g >= n) g -= n;
  return g;
}

// Principal square root of x + i y (branch cut on the negative real axis; the sign of a
// zero imaginary part selects the side, as in C99 csqrt), from the half-angle formulas
//   t = sqrt((|w| + |x|) / 2),  sqrt(w) = (t, y / (2t)) for x >= 0, (|y| / (2t), sign(y) t) else,
// with both square roots and the division taken from two reciprocal square roots:
// |w| = m rsqrt(m), m = x^2 + y^2, and with q = rsqrt((|w| + |x|)/2): t = ((|w| + |x|)/2) q,
// |y| / (2t) = |y| q / 2.  On GB300's narrow FP64 pipe this is about half the cost of hypot,
// sqrt and a division.  (m is formed without rescaling: |w| below ~1e-154 or above ~1e154
// in FP64 (1e-19 / 1e19 in FP32) loses accuracy, far outside the states of a diffusion run.)
// Reciprocal square root: CUDA's rsqrt in FP64; in FP32 the hardware approximation with
// subnormal inputs flushed to zero (rsqrt.approx.ftz: the same accuracy for normal inputs,
// without the subnormal handling; csqrt_principal keeps its inputs normal).
__device__ __forceinline__ double rsqrt_n(double a) { return rsqrt(a); }
__device__ __forceinline__ float rsqrt_n(float a) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}

template <class T>
__device__ __forceinline__ void csqrt_principal(T x, T y, T& rr, T& ri) {
  const T m = x * x + y * y;
  // w = 0, or in FP32 a modulus below ~1e-19 (m subnormal, which rsqrt.approx.ftz would take
  // as zero): sqrt(w) taken as (0, y)
  if (m == T(0) || (std::is_same<T, float>::value && m < T(1.17549435e-38f))) {
    rr = T(0);
    ri = y;
    return;
  }
  const T r = m * rsqrt_n(m);
  const T a = (r + fabs(x)) * T(0.5);
  const T q = rsqrt_n(a);
  const T t = a * q;
  const T h = T(0.5) * fabs(y) * q;
  if (x >= T(0)) {
    rr = t;
    ri = copysign(h, y);
  } else {
    rr = h;
    ri = copysign(t, y);
  }
}

// kappa(w) = 1 + c w^p for complex w = u + i v on the principal branch, 0^p = 0 (p > 0).
// p = 2.5 uses w^2 * sqrt(w); other exponents use the polar form |w|^p e^{i p arg w}.
template <class T>
__device__ __forceinline__ void kappa_power(T u, T v, T c, T p, T& kr, T& ki) {
  T wr = T(0), wi = T(0);
  if (u != T(0) || v != T(0)) {
    if (p == T(2.5)) {
      T sr, si;
      csqrt_principal<T>(u, v, sr, si);
      const T qr = u * u - v * v, qi = T(2) * u * v;
      wr = qr * sr - qi * si;
      wi = qr * si + qi * sr;
    } else {
      const T r = hypot(u, v), th = atan2(v, u);
      const T rp = pow(r, p);
      T sn, cs;
      sincos(p * th, &sn, &cs);
      wr = rp * cs;
      wi = rp * sn;
    }
  }
  kr = T(1) + c * wr;
  if constexpr (std::is_same<T, double>::value)
    ki = __dmul_rn(c, wi);  // (not for the caller to fuse with a sum, as below)
  else
    ki = c * wi;
}

// ---- double <-> float on the integer pipe ------------------------------------------------------
// On GB300 a conversion between double and float takes a slot of the FP64 pipe (2 lanes a clock per
// SM), the same as an FP64 addition; these do it with about ten and six integer instructions.  They
// return the bits of the hardware conversion (round to nearest even) whenever the value is zero or it
// and its float are normal, and set `slow` otherwise: the caller then redoes its conversions with
// narrow_hw / widen_hw in a loop that runs at most once, entered by a vote of the warp.  (A plain
// branch was turned into predicated conversions, which took the FP64 slots all the same: 217 us against
// 139 us for a MIXED kappa(u) pass on 160^3, 250 us with hardware conversions alone.)
__device__ __forceinline__ float narrow_fast(double d, bool& slow) {
  const unsigned hi = unsigned(__double2hiint(d)), lo = unsigned(__double2loint(d));
  const unsigned mag = hi & 0x7fffffffu;
  const bool zero = (mag | lo) == 0;               // (common: equal neighbours, zero imaginary parts)
  slow |= !zero && mag - (897u << 20) >= (254u << 20);  // exponent outside that of a normal float
  const unsigned v = __funnelshift_l(lo, hi, 3);   // exponent (9 low bits) and 23 mantissa bits
  const unsigned rem = lo << 3;                    // the 29 bits rounded away, at the top
  const unsigned half = 0x7fffffffu + (v & 1u);    // carries out of rem + half exactly when v rounds up
  const unsigned up = rem + half < half ? 1u : 0u;
  const unsigned m = zero ? 0u : v - (0x180u << 23) + up;
  return __uint_as_float(m | (hi & 0x80000000u));
}

__device__ __forceinline__ double widen_fast(float f, bool& slow) {
  const unsigned b = __float_as_uint(f), mag = b & 0x7fffffffu;
  const bool zero = mag == 0;
  slow |= !zero && mag - 0x00800000u >= 0x7f000000u;  // subnormal, infinite or not a number
  const unsigned hi = (zero ? 0u : (mag >> 3) + (896u << 20)) | (b & 0x80000000u);
  return __hiloint2double(int(hi), int(b << 29));
}

__device__ __forceinline__ float narrow_hw(double d) {
  float r;
  asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(r) : "d"(d));
  return r;
}
__device__ __forceinline__ double widen_hw(float f) {
  double r;
  asm volatile("cvt.f64.f32 %0, %1;" : "=d"(r) : "f"(f));
  return r;
}

// products that the compiler never fuses into a neighbouring add
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

// kappa(w) = 1 + c w^2.5 in float for a double state (MIXED), every rounding fixed: the formulas of
// csqrt_principal and kappa_power with |w|^2 and Re w^2 from rounded products and |w| + |x| fused.
__device__ __forceinline__ void kappa_power25_mixed(float x, float y, float c, float& kr, float& ki) {
  const float xx = __fmul_rn(x, x), yy = __fmul_rn(y, y), m = __fadd_rn(xx, yy);
  const float a = 0.5f * fmaf(m, rsqrt_n(m), fabsf(x)), q = rsqrt_n(a);
  const float t = __fmul_rn(a, q), h = __fmul_rn(0.5f * fabsf(y), q);
  float sr = x >= 0.f ? t : h, si = copysignf(x >= 0.f ? h : t, y);
  if (m < 1.17549435e-38f) {
    sr = 0.f;
    si = y;
  }
  const float qr = __fsub_rn(xx, yy), qi = __fmul_rn(2.f * x, y);
  const float wr = fmaf(qr, sr, -__fmul_rn(qi, si)), wi = fmaf(qr, si, __fmul_rn(qi, sr));
  kr = fmaf(c, wr, 1.f);
  ki = __fmul_rn(c, wi);
}

// ---- kappa(w) = 1 + c w^2.5, fewest operations ---------------------------------------------------
// With m = |w|^2, r = |w| = sqrt(m), b = r + |x| and q = 1 / sqrt(b):
//   sqrt(w) = (b q, |y| q) / sqrt(2) for x >= 0, the two swapped for x < 0, the sign of y on the
// imaginary part; the 1 / sqrt(2) goes into c, and w^2 = (m - 2 y^2, 2 x y).
//
// Square root and reciprocal square root in FP64 from one seed y0 (rsqrt.approx.ftz.f64) and one
// third-order Householder step: with e = 1 - a y0^2, 1/sqrt(a) = y0 (1 - e)^(-1/2) = y0 (1 + e/2 + 3 e^2/8 + ...),
// five FP64 instructions each; a normal and positive.
__device__ __forceinline__ double rsqrt_seed(double a) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  return r;
}
__device__ __forceinline__ double sqrt_h3(double a) {
  const double y = rsqrt_seed(a), t = a * y, e = fma(-t, y, 1.0);
  return fma(fma(0.375, e, 0.5), t * e, t);
}
__device__ __forceinline__ double rsqrt_h3(double a) {
  const double y = rsqrt_seed(a), t = a * y, e = fma(-t, y, 1.0);
  return fma(fma(0.375, e, 0.5), y * e, y);
}
__device__ __forceinline__ float sqrt_h3(float a) { return a * rsqrt_n(a); }
__device__ __forceinline__ float rsqrt_h3(float a) { return rsqrt_n(a); }

// |w|^2 kept normal (below, w^2.5 vanishes against 1 whatever its square root).  A NaN may come
// back as that or as itself; it reaches kappa(w) through x or y.
__device__ __forceinline__ double keep_normal(double m) {
  return __double2hiint(m) < 0x00100000 ? __hiloint2double(0x00100000, 0) : m;
}
__device__ __forceinline__ float keep_normal(float m) { return m < 1.17549435e-38f ? 1.17549435e-38f : m; }

template <class T>
__device__ __forceinline__ void kappa_power25_fast(T x, T y, T c, T& kr, T& ki) {
  const T yy = y * y, m = fma(x, x, yy);
  const T r = sqrt_h3(keep_normal(m));
  const T b = r + fabs(x), q = rsqrt_h3(b);
  const T t = b * q, h = fabs(y) * q;
  const T sr = x >= T(0) ? t : h;
  const T si = copysign(x >= T(0) ? h : t, y);
  const T qr = fma(x, x, -yy), qi = (x + x) * y;
  // (Which products are fused is written out, and ki is not for the caller to fuse with a sum: the same bits wherever
  // this is inlined.  An unrolled plane loop fused it in every other plane.)
  const T wr = fma(qr, sr, -mul_rn(qi, si)), wi = fma(qr, si, mul_rn(qi, sr));
  const T cs = c * T(0.70710678118654752440);  // loop-invariant
  kr = fma(cs, wr, T(1));
  ki = mul_rn(cs, wi);
}

// two floats to an instruction (sm_100 family)
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// kappa(w) = 1 + c w^2.5 of a pair; cs = c / sqrt(2)
__device__ __forceinline__ void kappa25_pair(float2 x, float2 y, float cs, float2& kr, float2& ki) {
  const float2 yy = mul2(y, y), m = fma2(x, x, yy);
  const float2 mc = make_float2(keep_normal(m.x), keep_normal(m.y));
  const float2 r = mul2(mc, make_float2(rsqrt_n(mc.x), rsqrt_n(mc.y)));
  const float2 b = make_float2(r.x + fabsf(x.x), r.y + fabsf(x.y));
  const float2 q = make_float2(rsqrt_n(b.x), rsqrt_n(b.y));
  const float2 t = mul2(b, q), h = make_float2(fabsf(y.x) * q.x, fabsf(y.y) * q.y);
  const bool p0 = x.x >= 0.f, p1 = x.y >= 0.f;
  const float2 sr = make_float2(p0 ? t.x : h.x, p1 ? t.y : h.y);
  const float2 si = make_float2(copysignf(p0 ? h.x : t.x, y.x), copysignf(p1 ? h.y : t.y, y.y));
  const float2 qr = fma2(make_float2(-2.f, -2.f), yy, m), nqr = mul2(make_float2(-1.f, -1.f), qr);
  const float2 nqi = mul2(mul2(make_float2(-2.f, -2.f), x), y);
  const float2 wr = fma2(nqi, si, mul2(qr, sr));
  const float2 nwi = fma2(nqi, sr, mul2(nqr, si));
  kr = fma2(make_float2(cs, cs), wr, make_float2(1.f, 1.f));
  ki = mul2(make_float2(-cs, -cs), nwi);
}

}  // namespace frkc2
