// Arithmetic of the scalar rules, shared by the replay kernels: tests on IEEE bits, integer
// powers, and divisions through a reciprocal.
#pragma once
#include <cuda_runtime.h>

#include "fmath.cuh"

namespace ndvm {

template <typename T> __device__ __forceinline__ T neg_zero() { return -(T)0; }

template <typename T> __device__ __forceinline__ T clamp_eps() { return (T)1e-8; }

// Tests on IEEE bit patterns run on the integer pipes, leaving the FP64 pipe to
// arithmetic (fbits keeps the compiler from turning them into FP64 compares).
// is_zero: +0 or -0.  gt_eps: x > 1e-8 with NaN false (IEEE order).
__device__ __forceinline__ bool is_zero(double x) { return (fbits(x) << 1) == 0; }
__device__ __forceinline__ bool is_zero(float x) { return x == 0.0f; }
__device__ __forceinline__ bool gt_eps(double x) {
  const long long b = fbits(x);
  return b > __double_as_longlong(1e-8) && (b & 0x7fffffffffffffffLL) <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool gt_eps(float x) {
  const int b = __float_as_int(x);
  return b > __float_as_int(1e-8f) && (b & 0x7fffffff) <= 0x7f800000;
}

// x with its sign bit flipped when neg is set (IEEE negation, exact for every value)
__device__ __forceinline__ double flip_sign(double x, unsigned neg) {
  return __longlong_as_double(fbits(x) ^ ((long long)neg << 63));
}
__device__ __forceinline__ float flip_sign(float x, unsigned neg) {
  return __int_as_float(__float_as_int(x) ^ (int)(neg << 31));
}

// a^n by left-to-right repeated multiplication, and n a^(n-1) (the base adjoint of an
// integer power): small n take straight-line code with literal factors (a loop with a
// run-time trip count compiles to predicated multiplies, and converting n to a float
// costs an FP64 slot); the same operations in the same order either way
template <typename T> __device__ __forceinline__ T powi_loop(T a, int n) {
  T z = a;
#pragma unroll 1
  for (int i = 1; i < n; i++) z = z * a;
  return z;
}
template <typename T> __device__ __forceinline__ T powi_rep(T a, int n) {
  switch (n) {
    case 0: return (T)1;
    case 1: return a;
    case 2: return a * a;
    case 3: return (a * a) * a;
    case 4: return ((a * a) * a) * a;
    default: return powi_loop(a, n);
  }
}
template <typename T> __device__ __forceinline__ T powi_deriv(T a, int n) {  // n >= 1
  switch (n) {
    case 1: return (T)1 * (T)1;
    case 2: return (T)2 * a;
    case 3: return (T)3 * (a * a);
    case 4: return (T)4 * ((a * a) * a);
    default: return (T)n * powi_loop(a, n - 1);
  }
}

// correctly rounded reciprocal: the value of the IEEE division 1 / x, at lower cost
__device__ __forceinline__ double rcp_rn(double x) { return __drcp_rn(x); }
__device__ __forceinline__ float rcp_rn(float x) { return __frcp_rn(x); }

// a / b from r, the correctly rounded reciprocal of b, by one correction step
// (Markstein): q = a r, e = a - b q (exact by fma), q + r e.  The step is taken where a,
// b and the quotient lie well inside the normal range (exponents within +-500 for double,
// +-60 for float, zeros, infinities and NaNs excluded); elsewhere the IEEE division.
__device__ __forceinline__ bool div_step_ok(double a, double b) {
  const unsigned ea = (unsigned)(fbits(a) >> 52) & 0x7ffu;
  const unsigned eb = (unsigned)(fbits(b) >> 52) & 0x7ffu;
  return ea - 523u <= 1000u && eb - 523u <= 1000u;
}
__device__ __forceinline__ bool div_step_ok(float a, float b) {
  const unsigned ea = (__float_as_uint(a) >> 23) & 0xffu, eb = (__float_as_uint(b) >> 23) & 0xffu;
  return ea - 67u <= 120u && eb - 67u <= 120u;
}
// the IEEE division and the correctly rounded reciprocal as calls (rarely taken paths;
// see fmath.cuh's slow paths)
template <typename T> __device__ __noinline__ T slow_div(T a, T b) { return a / b; }
template <typename T> __device__ __noinline__ T slow_rcp(T b) { return rcp_rn(b); }

// 1/b for b with an exponent within +-500 (div_step_ok): the hardware estimate
// (rcp.approx.ftz.f64, off the FP64 pipe, more than 20 correct bits) refined by one third-order
// step, y + y (e + e^2) with e = 1 - b y, which triples them; 3 FP64 instructions (two
// Newton steps take 4) and no special-case code.  The result is within a hair of half an ulp, which is what the
// correction step of a division needs.
__device__ __forceinline__ double rcp_newton(double b) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(b));
  const double e = fma(-b, y, 1.0);
  return fma(y, fma(e, e, e), y);
}
__device__ __forceinline__ float rcp_newton(float b) { return __frcp_rn(b); }

// a / b and 1/b (into *r): in the safe range by the Newton reciprocal and one correction
// step, else the IEEE division and the correctly rounded reciprocal
template <typename T>
__device__ __forceinline__ T div_rcp(T a, T b, T* r);
template <typename T>
__device__ __forceinline__ T div_rcp_q(T a, T b) {  // a / b alone
  T r;
  return div_rcp(a, b, &r);
}
template <typename T>
__device__ __forceinline__ T div_rcp(T a, T b, T* r) {
  if (!div_step_ok(a, b)) {
    *r = slow_rcp(b);
    return slow_div(a, b);
  }
  const T y = rcp_newton(b);
  *r = y;
  const T q = a * y;
  return fma(y, fma(-b, q, a), q);
}
template <typename T>
__device__ __forceinline__ T div_by_rcp(T a, T b, T r) {
  if (!div_step_ok(a, b)) return slow_div(a, b);
  const T q = a * r;
  return fma(r, fma(-b, q, a), q);
}

}  // namespace ndvm
