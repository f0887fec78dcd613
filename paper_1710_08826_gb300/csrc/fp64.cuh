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

// 1 / x for any x: the step above where x and 1 / x are normal (tested on the integer pipe), else a
// division.
__device__ __forceinline__ double recip(double x) {
  const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
  return h - 0x00300000u < 0x7fa00000u - 0x00300000u ? rcp64(x) : 1.0 / x;
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

// ---------------------------------------------------------------------------------------
// exp and erfcx from tables.  Tables are read from shared memory, whose lookups (and bank
// conflicts) cost nothing next to a 16-cycle FP64 slot, and the table index is formed on the
// integer and FP32 pipes, so that only the polynomial is left on the FP64 pipe.
// The tables are computed on the host (fp64.cu) in extended precision.  Largest difference from CUDA's
// functions over 16M arguments: exp_tab 1 unit of the last place (1.5 where |x| nears 700), herfcx_tab 2, rcp64 half a unit.
// ---------------------------------------------------------------------------------------
constexpr int kExpTab = 2048;       // 2^(j / 2048)
constexpr int kErfcxStep = 32;      // nodes of erfcx per unit of its argument
constexpr int kErfcxMax = 6;        // table range [0, 6]
constexpr int kErfcxTab = kErfcxStep * kErfcxMax + 1;
constexpr int kErfcxDeg = 7;

constexpr int kLogTab = 1024;

struct alignas(16) ErfcxTable {
  double node[kErfcxTab];                 // i / 32
  double herfcx[kErfcxDeg + 1][kErfcxTab];  // erfcx(node + r) / 2 = sum_d herfcx[d][i] r^d, |r| <= 1 / 64
};
struct alignas(16) ExpTable {
  double exp2j[kExpTab];
};
struct alignas(16) LogTable {
  double inv[kLogTab], ref[kLogTab];  // about 1 / (1 + (j + 1/2) / 1024), and minus its logarithm
};
struct Fp64Tables {
  ErfcxTable erfcx;
  ExpTable exp;
  LogTable log;
};
// What a kernel keeps in shared memory: the functions that it calls.
struct TimeTables {
  ErfcxTable erfcx;
  ExpTable exp;
};
struct SopTables {
  ExpTable exp;
  LogTable log;
};

// The block's copy of a table (no barrier after).
template <typename Table>
__device__ __forceinline__ void load_table(Table& s, const Table& g) {
  static_assert(sizeof(Table) % sizeof(double2) == 0, "16-byte pieces");
  for (int i = threadIdx.x; i < (int)(sizeof(Table) / sizeof(double2)); i += blockDim.x)
    reinterpret_cast<double2*>(&s)[i] = __ldg(reinterpret_cast<const double2*>(&g) + i);
}
__device__ __forceinline__ void load_fp64_tables(TimeTables& s, const Fp64Tables* __restrict__ g) {
  load_table(s.erfcx, g->erfcx);
  load_table(s.exp, g->exp);
}
__device__ __forceinline__ void load_fp64_tables(SopTables& s, const Fp64Tables* __restrict__ g) {
  load_table(s.exp, g->exp);
  load_table(s.log, g->log);
}

// |x| (x normal, 2^-126 <= |x| < 2^128) as a float, truncated, without the FP64 pipe: the exponent
// rebiased and the mantissa's top 23 bits.  Smaller arguments give some tiny or negative float; the
// callers use it only to pick a table entry.
__device__ __forceinline__ float abs_float_trunc(double x) {
  const int h = __double2hiint(x) & 0x7fffffff;
  const int f = ((h - (896 << 20)) << 3) | ((unsigned)__double2loint(x) >> 29);
  return h < (897 << 20) ? 0.f : __int_as_float(f);
}

// exp(x), table-driven (P. T. P. Tang, ACM TOMS 15 (1989) 144): x = n ln2 / 2048 + r, exp(x) = 2^(n / 2048) exp(r)
// with n / 2048 split into an exponent and a table index, |r| <= ln2 / 4096 = h and a degree-3 polynomial
// (the series with its r^4 replaced by h^2 r^2, which leaves h^4 / 192 = 4e-18): 7 slots of the FP64
// pipe and within one unit of the last place, where exp() takes about twenty.  |x| > 704 (and NaN) goes
// to exp().  A table of 256 entries needs degree 4.
__device__ __forceinline__ double exp_tab(double x, const ExpTable& tab) {
  const int hx = __double2hiint(x);
  if ((hx & 0x7fffffff) >= 0x40860000) return exp(x);
  const float f = abs_float_trunc(x) * 2954.639443740597f;  // 2048 / ln 2
  const int na = __float2int_rn(f), n = hx < 0 ? -na : na;
  // n as a double: 2^52 + 2^51 + n holds n in its low word
  const double dn = __hiloint2double(0x43380000 + (n >> 31), n) - 6755399441055744.0;
  // ln2 / 2048 as a 31-bit head (n times it is exact) and the rest
  double r = ::fma(dn, -0.0003384507717782981, x);
  r = ::fma(dn, 2.0512280628325608e-14, r);
  const double p = ::fma(r, 1.0 / 6.0, 0.500000001193218);  // 1/2 + h^2 / 24
  const double q = ::fma(r * r, p, r);
  const double t = tab.exp2j[n & (kExpTab - 1)];
  const double s = __hiloint2double(__double2hiint(t) + ((n >> 11) << 20), __double2loint(t));
  return ::fma(s, q, s);
}

// log(x) for x > 0, table-driven (P. T. P. Tang, ACM TOMS 16 (1990) 378): x = 2^e m, j the top 10 bits of m's
// fraction, r = m inv_j - 1 with |r| < 2^-10.9, log x = e ln2 - log inv_j + log1p(r) with log1p to degree 4
// (truncation 8e-18): 8 slots, the error about one unit of the last place of e ln2 - log inv_j (so
// absolute, not relative, for x near 1), where log() takes some twenty-five.  Subnormal, infinite and NaN
// arguments go to log().
__device__ __forceinline__ double log_tab(double x, const LogTable& tab) {
  if (!positive_normal(x)) return log(x);
  const int hx = __double2hiint(x);
  const int j = (hx >> 10) & (kLogTab - 1), e = (hx >> 20) - 1023;
  const double m = __hiloint2double((hx & 0x000fffff) | 0x3ff00000, __double2loint(x));
  const double r = ::fma(m, tab.inv[j], -1.0);
  const double de = __hiloint2double(0x43380000 + (e >> 31), e) - 6755399441055744.0;
  double p = ::fma(r, -0.25, 1.0 / 3.0);
  p = ::fma(r, p, -0.5);
  const double q = ::fma(r * r, p, r);
  return ::fma(de, 0.693147180559945309417, tab.ref[j]) + q;
}

// erfcx(u) / 2 for 0 <= u < 6: the degree-7 interpolant of the nearest node (relative error of the
// interpolation below 1e-17), 8 slots.
__device__ __forceinline__ double herfcx_tab(double u, const ErfcxTable& tab) {
  const int i = __float2int_rn(abs_float_trunc(u) * (float)kErfcxStep);
  const double r = u - tab.node[i];
  double p = tab.herfcx[kErfcxDeg][i];
#pragma unroll
  for (int d = kErfcxDeg - 1; d >= 0; --d) p = ::fma(p, r, tab.herfcx[d][i]);
  return p;
}

// The same interpolants of erfcx(u) / 2 in FP32: degree 3 (error of the interpolation 4e-9).
constexpr int kErfcxDeg32 = 3;
struct Fp32Tables {
  float herfcx[kErfcxDeg32 + 1][kErfcxTab];
};

#ifndef __CUDACC_RTC__
// The context's device copies of the tables, built on first use (host pointer arithmetic only
// afterwards) and freed with the context.
int fp64_tables(goo_ctx* ctx, const Fp64Tables** dev);
int fp32_tables(goo_ctx* ctx, const Fp32Tables** dev);
#endif

}  // namespace goo
