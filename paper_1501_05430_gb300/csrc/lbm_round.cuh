// lbm_round.cuh -- FP32 quotients and square roots of lane pairs, quotients by small
// integers and quotients that share a divisor, each with the bits of the IEEE
// operation.  For units compiled with -fmad=false.
#pragma once

#include <cuda_runtime.h>
#include <math.h>

namespace lbm_round {

// F2 holds two nodes of a row; its operations are the packed FP32 instructions,
// each lane rounded like the scalar operation.
struct F2 {
  float2 v;
};
// The assembler joins a packed product and the packed sum it goes into to one
// fused operation whatever their rounding modifiers say, so sums are written as
// fused operations themselves, a * 1 + b with a factor that it cannot know.
static __constant__ float2 c_one = {1.0f, 1.0f}, c_minus = {-1.0f, -1.0f};
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return {__ffma2_rn(a.v, c_one, b.v)}; }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return {__ffma2_rn(b.v, c_minus, a.v)}; }
__device__ __forceinline__ F2 operator-(F2 a) { return {__ffma2_rn(a.v, c_minus, make_float2(-0.0f, -0.0f))}; }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ F2 operator/(F2 a, F2 b) { return {make_float2(a.v.x / b.v.x, a.v.y / b.v.y)}; }
__device__ __forceinline__ F2 vfma(F2 a, F2 b, F2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ F2 both(float c) { return {make_float2(c, c)}; }

template <class V>
struct Val;
template <>
struct Val<double> {
  typedef double R;
  static constexpr int N = 1;
  __device__ __forceinline__ static double bc(double c) { return c; }
  __device__ __forceinline__ static double lane(double v, int) { return v; }
  __device__ __forceinline__ static void set(double &v, int, double x) { v = x; }
};
template <>
struct Val<float> {
  __device__ __forceinline__ static float bc(float c) { return c; }
};
template <>
struct Val<F2> {
  typedef float R;
  static constexpr int N = 2;
  __device__ __forceinline__ static F2 bc(float c) { return {make_float2(c, c)}; }
  __device__ __forceinline__ static float lane(F2 v, int k) { return k ? v.v.y : v.v.x; }
  __device__ __forceinline__ static void set(F2 &v, int k, float x) { (k ? v.v.y : v.v.x) = x; }
};

// ---- corrected approximations ---------------------------------------------------
// Markstein (IBM J. Res. Dev. 34, 1990): with y = 1/b rounded to nearest and q
// within one last place of a/b, q + y (a - b q) is a/b rounded to nearest, and
// a - b q is exact, as long as nothing leaves the normal range.  y comes from the
// hardware's approximation by one correction (compared with 1/b for every b in
// [2^-40, 2^40]); a y is within two last places of a/b, a first correction brings
// it within one and a second one makes it exact.
// plain, in_range: the operands for which that holds, b in [2^-40, 2^40] and |a| in
// [2^-80, 2^40] or 0: the quotient lies between 2^-120 and 2^80 and the remainder's
// last place at 2^-126 or above.  Any others are divided by the division.  The one
// difference left is the sign of a quotient of 0.

// 2 |x| - 1 as an integer: ordered like |x|, but 0 comes last
__device__ __forceinline__ unsigned key(float x) { return 2u * __float_as_uint(x) - 1u; }
__device__ __forceinline__ bool in_range(F2 a, F2 c) {
  const unsigned least = min(min(key(a.v.x), key(a.v.y)), min(key(c.v.x), key(c.v.y)));
  const float most = fmaxf(fmaxf(fabsf(a.v.x), fabsf(a.v.y)), fmaxf(fabsf(c.v.x), fabsf(c.v.y)));
  return least >= 2u * ((127u - 80u) << 23) - 1u && most <= 0x1p40f;  // (NaN stays NaN)
}

struct Reciprocal {
  F2 nb, y;
  __device__ __forceinline__ explicit Reciprocal(F2 b) : nb(-b) {
    float x, z;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(x) : "f"(b.v.x));
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(z) : "f"(b.v.y));
    y = {make_float2(x, z)};
    y = vfma(vfma(nb, y, both(1.0f)), y, y);
  }
  __device__ __forceinline__ F2 under(F2 a) const {  // (+0 for -0)
    const F2 q = a * y, q1 = vfma(vfma(nb, q, a), y, q);
    return vfma(vfma(nb, q1, a), y, q1);
  }
};

// a / b and c / b; plain: the caller knows that b is in range.
__device__ __forceinline__ void quotients(F2 a, F2 c, F2 b, bool plain, F2 &qa, F2 &qc) {
  const Reciprocal r(b);
  qa = r.under(a), qc = r.under(c);
  if (__builtin_expect(!(plain && in_range(a, c)), 0)) qa = a / b, qc = c / b;
}
__device__ __forceinline__ void quotients(double a, double c, double b, bool, double &qa, double &qc) {
  qa = a / b, qc = c / b;
}

// sqrt(max(0, a)).
__device__ __forceinline__ F2 root0(F2 a) { return {make_float2(sqrtf(fmaxf(0.0f, a.v.x)), sqrtf(fmaxf(0.0f, a.v.y)))}; }
__device__ __forceinline__ double root0(double a) { return sqrt(fmax(0.0, a)); }
__device__ __forceinline__ float root0(float a) { return sqrtf(fmaxf(0.0f, a)); }
// The same for a <= 0 or in [2^-80, 2^40].  One coupled Newton step for sqrt and
// 1/(2 sqrt) from the hardware's approximation of the latter, and a last one with
// the exact remainder (Markstein, as above; compared with the square root for every
// a in that range).
__device__ __forceinline__ F2 root0_in_range(F2 a) {
  const float x = fmaxf(0.0f, a.v.x), z = fmaxf(0.0f, a.v.y);
  float yx, yz;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yx) : "f"(fmaxf(x, 1.17549435e-38f)));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yz) : "f"(fmaxf(z, 1.17549435e-38f)));
  const F2 s = {make_float2(x, z)}, y = {make_float2(yx, yz)}, g = s * y, nh = both(-0.5f) * y;
  const F2 e = vfma(nh, g, both(0.5f)), g1 = vfma(g, e, g), nh1 = vfma(nh, e, nh);
  return vfma(vfma(g1, g1, -s), nh1, g1);
}

// x / d for d = 3, 6, 9, 12, 36, correctly rounded, from 1/d = h + l (Brisebarre,
// Muller, Raina, "Accelerating correctly rounded floating-point division when
// the divisor is known in advance", IEEE Trans. Computers 53, 2004).  Before its
// rounding x h + RN(x l) is within 2^-2p (relative; p = 53 or 24) of x / d, and
// x / d, whose odd denominator part is 3 or 9, is never nearer than 1/18 of a
// last place to a midpoint between two numbers.  x finite, and 0 (the result's
// sign aside) or so large that x l is a normal number (FP32: |x| >= 2^-94).
template <class R>
inline void const_reciprocal(R d, R *h, R *l) {
  *h = (R)1 / d;
  *l = (R)fma(-d, *h, (R)1) / d;  // the remainder is exact
}
template <class V, class R>
__device__ __forceinline__ V div_const(V x, R h, R l) {
  return vfma(x, Val<V>::bc(h), x * Val<V>::bc(l));
}

// a / b from y = 1/b rounded to nearest by two corrections, as Reciprocal::under, in
// FP32 or FP64 (five instructions where several quotients share a divisor).  Finite
// operands in the normal range; a below 1e-30 in FP32 (its remainder leaves the normal
// range) may be a last place off.
template <typename R>
__device__ __forceinline__ R quot(R a, R b, R y) {
  const R q0 = a * y, q1 = vfma(vfma(-b, q0, a), y, q0);
  return vfma(vfma(-b, q1, a), y, q1);
}
// a / N for a small integer N, for such a: in FP32 one correction is enough for 3, 9
// and their multiples by powers of two (compared for every significand).
template <int N, typename R>
__device__ __forceinline__ R over(R a) {
  constexpr R y = (R)1 / (R)N;
  if constexpr ((N & (N - 1)) == 0) return a * y;
  if constexpr (sizeof(R) == 8) return quot(a, (R)N, y);
  const R q = a * y;
  return vfma(vfma(-(R)N, q, a), y, q);
}

}  // namespace lbm_round
