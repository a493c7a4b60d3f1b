// fp64_math.cuh -- double division and square root for the FP64-bound kernels.
//
// GB300 does 2 double operations per SM and clock, so kernels in double are
// bound by the number of double instructions alone (integer and FP32 ones
// are nearly free beside them).  The functions here spend 6 of them on a
// quotient (3 on a further one by the same divisor) and 8 on a square root:
// an approximate reciprocal (rcp.approx / rsqrt.approx, about 20 bits), one
// third-order Newton step on it, and the final correction by the exact
// residual of P. Markstein ("Computation of elementary functions on the IBM
// RISC System/6000", IBM J. Res. Dev. 34, 1990): with a reciprocal good to an
// ulp the corrected result is the correctly rounded one, as IEEE division and
// square root give it (tests/test_gpu_fp64_math.py: no mismatch against them in
// 2^30 random operands of each, 2^30 next to a tie, and the edges of the ranges).
//
// They hold where nothing under- or overflows on the way: the *_raw forms
// leave the check to the caller, the others test the exponents with integer
// operations and take the IEEE operator outside.
#pragma once

#include <cuda_runtime.h>

namespace shasta {
namespace f64 {

__device__ __forceinline__ int hi(double x) { return __double2hiint(x); }
// exponent field and top mantissa bits of |x|
__device__ __forceinline__ unsigned mag(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }
__device__ __forceinline__ bool is_zero(double x) { return (mag(x) | (unsigned)__double2loint(x)) == 0u; }
// |x| in [2^lo, 2^hi)
template <int LO, int HI>
__device__ __forceinline__ bool within(double x) {
  return mag(x) - (unsigned)((LO + 1023) << 20) < (unsigned)((HI - LO) << 20);
}
// x 2^k for normal x and result
template <int K>
__device__ __forceinline__ double scale(double x) {
  return __hiloint2double(hi(x) + (K << 20), __double2loint(x));
}

__device__ __forceinline__ long long bits(double x) { return __double_as_longlong(x); }

// float -> double and back by the bit patterns (the conversion instructions
// go through the double pipe: one of its slots each).  Zeros and normal
// numbers; the rest, and what rounds to a subnormal float, by the instruction
// (out of line: inlined, the compiler predicates it and every cell pays).
static __device__ __noinline__ double widen_rest(float f) { return (double)f; }
static __device__ __noinline__ float narrow_rest(double x) { return (float)x; }
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u || a == 0u)
    return __hiloint2double((int)((u & 0x80000000u) | (a ? (a >> 3) + 0x38000000u : 0u)), (int)(u << 29));
  return widen_rest(f);
}
__device__ __forceinline__ double widen(double x) { return x; }
template <class T>
__device__ __forceinline__ T narrow(double x) {
  if constexpr (sizeof(T) == 8) {
    return x;
  } else {
    const unsigned a = mag(x);
    const unsigned long long b = (unsigned long long)bits(x) & 0x7fffffffffffffffull;
    const bool z = is_zero(x);
    if (a - 0x38100000u < 0x47e00000u - 0x38100000u || z) {  // 2^-126 <= |x| < 2^127, or zero
      const unsigned long long r = b + 0x0fffffffull + ((b >> 29) & 1ull);  // to nearest even
      const unsigned f = z ? 0u : (unsigned)(r >> 29) - (896u << 23);
      return __uint_as_float(f | ((unsigned)hi(x) & 0x80000000u));
    }
    return narrow_rest(x);
  }
}

// 1/y to about an ulp, y normal and well inside the range.  For a
// significand of ones the quotients of the correction below can be ties that
// only the rounded-up reciprocal breaks the right way: there r is a power of
// two and takes its last bit.
__device__ __forceinline__ double recip_raw(double y) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(y));
  const double e = fma(-y, r, 1.0);
  r = fma(r, fma(e, e, e), r);
  const bool ones = ((hi(y) | 0xfff00000) & __double2loint(y)) == -1;
  return __hiloint2double(hi(r), __double2loint(r) | (ones ? 1 : 0));
}
// a/y from r = recip_raw(y).
__device__ __forceinline__ double quot_raw(double a, double y, double r) {
  const double q = a * r;
  return fma(fma(-y, q, a), r, q);
}
__device__ __forceinline__ double sqrt_raw(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double g = x * y;
  const double e = fma(-g, y, 1.0);
  const double p = e * fma(0.375, e, 0.5);
  const double g1 = fma(g, p, g);            // sqrt(x)
  const double h = scale<-1>(fma(y, p, y));  // 1 / (2 sqrt(x))
  return fma(fma(-g1, g1, x), h, g1);
}

// the IEEE operators, out of line: inlined, the compiler predicates them and
// every cell pays
static __device__ __noinline__ double ieee_div(double a, double y) { return a / y; }
static __device__ __noinline__ double ieee_sqrt(double x) { return ::sqrt(x); }

__device__ __forceinline__ double div(double a, double y) {
  if (within<-400, 400>(y) && (within<-500, 500>(a) || is_zero(a))) {
    const double r = recip_raw(y);
    const double q = a * r;
    return is_zero(a) ? q : fma(fma(-y, q, a), r, q);
  }
  return ieee_div(a, y);
}
__device__ __forceinline__ double sqrt(double x) {
  if (hi(x) > 0 && within<-900, 1000>(x)) return sqrt_raw(x);
  return ieee_sqrt(x);
}

}  // namespace f64
}  // namespace shasta
