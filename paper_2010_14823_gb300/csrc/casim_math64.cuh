// FP64 functions and quotients of the FP64 form, whose FP64 pipe issues one
// instruction per SM every ~19 cycles while the integer pipe idles.
//
// exp and log are CUDA's, called out of line: inlined at every use, the
// processes' code does not fit the instruction cache (256x256x100 stratus 6.0 ms
// out of line, 8.0 inlined; deep convection 10.6 and 12.6).  Table-driven ones of
// fewer operations took 4.9 and 8.7 ms, but a field's distance from the formulas
// evaluated in 64 bits was 3.1e-15 with them, 7e-16 with CUDA's: not used.
// A quotient takes 6 FP64 operations and has the bits of the division, its range checks on
// the integer pipe: the hardware's reciprocal estimate (relative error ~2^-20),
// one third-order step 1/b = r (1 + e + e^2 + ..), e = 1 - b r, and Markstein's
// final correction (IBM J. Res. Dev. 34, 1990) by the remainder a - q b, which
// a fused multiply-add gives exactly.  Operands outside the ranges below take
// the division itself.
#pragma once

#include <cuda_runtime.h>

namespace casim_dev {

static __device__ __noinline__ double exp64(double x) { return ::exp(x); }
static __device__ __noinline__ double log64(double x) { return ::log(x); }
static __device__ __noinline__ double div64_general(double a, double b) { return a / b; }

// exponent well inside the range: 2^-511 <= |x| < 2^511
__device__ __forceinline__ bool div64_range(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) - 0x20000000u < 0x3fe00000u;
}

// The one exception to the correction's rounding theorem is a divisor whose
// mantissa is all ones: divisors whose low word is take the division.
__device__ __forceinline__ bool div64_divisor(double b) {
  return div64_range(b) && (unsigned)__double2loint(b) != 0xffffffffu;
}

// 1/b, for b inside that range
__device__ __forceinline__ double rcp64(double b) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
  const double e = fma(-b, r, 1.0);
  return fma(fma(e, e, e), r, r);
}

// a / b from r = 1/b for a divisor as above; a outside the range (but for zero)
// takes the division
__device__ __forceinline__ double div64_by(double a, double b, double r) {
  const bool za = (((unsigned)__double2hiint(a) & 0x7fffffffu) | (unsigned)__double2loint(a)) == 0u;
  if (!za && !div64_range(a)) return div64_general(a, b);
  const double q = a * r;
  return za ? q : fma(fma(-b, q, a), r, q);   // (zero: q has the sign)
}

__device__ __forceinline__ double div64(double a, double b) {
  if (!div64_divisor(b)) return div64_general(a, b);
  return div64_by(a, b, rcp64(b));
}

// several quotients of one divisor
struct Div64 {
  double b = 1.0, r = 1.0;
  bool in_range = true;
  Div64() = default;
  __device__ __forceinline__ explicit Div64(double d) : b(d), r(rcp64(d)), in_range(div64_divisor(d)) {}
  __device__ __forceinline__ double operator()(double a) const {
    return in_range ? div64_by(a, b, r) : div64_general(a, b);
  }
};

}  // namespace casim_dev
