// fp64.cuh -- FP64 arithmetic for the plain-precision kernels, written around GB300's FP64 pipe.
//
// The pipe retires 2 lanes per SM and cycle (1/64 of FP32): one warp instruction occupies it
// for 16 cycles.  FP64 additions, multiplications, comparisons and conversions from or to FP64
// all take such a slot (measured: 490 to 580 G lanes/s each in a short kernel), while integer
// and FP32 instructions and the approximate FP64 reciprocal of the special-function unit (rcp.approx.ftz.f64: 4180
// G/s) issue beside it for nothing.  The FP64 kernels are bound by the number of slots per event, so
// these helpers move sign and range tests, exponents and seeds to the other pipes.
#pragma once

#include "common.cuh"

namespace goo {

// 1 / x for a normal x by one third-order step (y + y (e + e^2), e = 1 - x y: the geometric series
// cut after its second term) from the special-function unit's approximation, whose residual e
// is below 2^-20 (measured 9.4e-7): three FMAs, the result within 2^-53 of 1 / x.  Where the
// approximation leaves the normal range (|x| below 2^-1022 or above 2^1022) the result is as
// undefined as the seed; the callers keep such arguments away.
__device__ __forceinline__ double rcp64(double x) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = ::fma(-x, y, 1.0);
  return ::fma(y, ::fma(e, e, e), y);
}

// True for a positive, normal, finite x: one integer test on the high word (a comparison of
// doubles takes a slot of the FP64 pipe).
__device__ __forceinline__ bool positive_normal(double x) {
  return (unsigned)(__double2hiint(x) - 0x00100000) < 0x7fe00000u;
}

// Sum of log(s_i) as the logarithm of the product: sum log s_i = log(prod m_i) + ln 2 sum e_i
// with s_i = m_i 2^e_i.  A factor costs one multiplication on the FP64 pipe (the exponents are
// split off with integer instructions) where log() takes some twenty-five slots, and it is
// the more accurate form: each factor is rounded once, relative, where a logarithm was
// rounded to its own last place and again when it was added to the running sum.
struct LogProduct {
  double m = 1.0;  // product of the mantissas, in [1, 2)
  int e = 0;       // sum of the exponents
  // x: positive and normal (positive_normal)
  __device__ __forceinline__ void mul(double x) {
    const int hx = __double2hiint(x);
    const double p = m * __hiloint2double((hx & 0x000fffff) | 0x3ff00000, __double2loint(x));  // in [1, 4)
    const int hp = __double2hiint(p);
    e += (hx >> 20) + (hp >> 20) - 2 * 1023;
    m = __hiloint2double((hp & 0x000fffff) | 0x3ff00000, __double2loint(p));
  }
  __device__ __forceinline__ double log_value() const { return ::fma((double)e, 0.693147180559945309417, log(m)); }
};

}  // namespace goo
