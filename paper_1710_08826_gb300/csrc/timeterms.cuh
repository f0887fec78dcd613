// timeterms.cuh -- decay-time machinery shared by the time-dependent amplitude models
// (td4.cu: four-body; dalitz.cu: three-body): the Faddeeva function w(z) (Weideman's
// rational approximation, J. A. C. Weideman, SIAM J. Numer. Anal. 31 (1994) 1497; host and
// device), the convolution E(g; t, s) of e^{-g t'} (t' >= 0) with a Gaussian resolution for
// real and complex g, and the mixing terms with their derivatives.  The formulas are stated
// at the top of td4.cu.
//
// The rate needs the four terms only through
//   R = |A|^2 P + |B|^2 Q + Re(A B*) T_sh + Im(A B*) T_s,
//   P = (T_ch + T_c)/2,  Q = (T_ch - T_c)/2,
// i.e. the convolutions of e^{-G t'} [cosh(y G t') +- cos(x G t')]/2, e^{-G t'} sinh(y G t')
// and e^{-G t'} sin(x G t').  For small mixing Q, T_sh and T_s are tiny differences of nearly
// equal convolved exponentials (Q = O(x^2 + y^2), T_sh = O(y)): formed as such differences in
// FP32 they keep only a few significant digits.  Where
// z = max(|x|, |y|) G (max(t, 0) + 6 s) is small they are therefore summed as power series in
// the moments of the resolution-convolved exponential,
//   M_n(t) = int_0^inf t'^n e^{-G t'} N(t - t'; 0, s) dt',  w_n = G^n M_n,
//   P = sum_m a_m w_2m,  Q = sum_m b_m w_2m,  T_sh = sum_m y^(2m+1) / (2m+1)! w_(2m+1),
//   T_s = sum_m (-1)^m x^(2m+1) / (2m+1)! w_(2m+1),
//   a_m, b_m = (y^2m +- (-1)^m x^2m) / (2 (2m)!),
// from the Taylor series of cosh and cos, with every term of one sign for t > G s^2.  The
// moments follow from M_0 = E(G) (one erfcx) by the recurrence obtained by integrating
// t' N(t - t') by parts,
//   w_1 = G (v M_0 + s^2 N(t)),  w_(n+1) = G v w_n + n G^2 s^2 w_(n-1),  v = t - G s^2.
// Elsewhere (large mixing) the terms come from the Faddeeva path, where the differences are
// not small.
//
// Derivatives.  The four functions f = e^{-G t'} (...) are closed under d / d t',
//   f_P'  = -G f_P + G (y f_sh - x f_s)/2,   f_Q' = -G f_Q + G (y f_sh + x f_s)/2,
//   f_sh' = -G f_sh + G y (f_P + f_Q),       f_s' = -G f_s + G x (f_P - f_Q),
// with f_P(0) = 1 and the others 0 there, so every derivative of the terms is a combination of
// the terms themselves; no series is summed for it.  Integrating t' N(t - t') by parts once
// more, the convolutions C_f of t' f(t') are
//   C_P  = v P + s^2 N(t) + s^2 G (y T_sh - x T_s)/2,  C_Q = v Q + s^2 G (y T_sh + x T_s)/2,
//   C_sh = v T_sh + s^2 G y (P + Q),                   C_s = v T_s + s^2 G x (P - Q),
// and for the event's weights (|A|^2, |B|^2, Re AB*, Im AB*) = (a, b, r, i)
//   dR/dx = G X,  X = (b - a)/2 C_s + i (C_P - C_Q),
//   dR/dy = G Y,  Y = (a + b)/2 C_sh + r (C_P + C_Q),
//   G dR/dG = -G Z + G (y Y + x X),  Z = a C_P + b C_Q + r C_sh + i C_s   (G d f / d G = t' f'),
//   dR/ds = s d^2 R / dt^2   (heat equation of the Gaussian)
//         = s [G^2 (R - 2 (y E_y + x E_x) + y^2 R_y - x^2 R_x) + N(t) (G (y r + x i - a) - t a / s^2)],
//   E_y = (a + b)/2 T_sh + r T_ch,  E_x = (b - a)/2 T_s + i T_c,
//   R_y = (a + b)/2 T_ch + r T_sh,  R_x = (a - b)/2 T_c + i T_s.
// The lanes per event are X, Y, Z and the bracket without its G^2 R, each over R; the last block
// applies the constant factors (time_gradient).  The kernels are bound by their instructions (FP32)
// or FP64 slots: summing the derivatives as series too and branching between two erfcx calls cost
// 2M events FP32 64.1 us (four-body) and 114.5 us (three-body), this 59.3 and 97.3 us; 1M events
// FP64 four-body 1222 us, this 872 us (the kernels' later figures stand beside them).
#pragma once

#include <cmath>
#include <vector>

#include "common.cuh"
#include "fp64.cuh"

namespace goo {

constexpr int kWMax = 40;
constexpr int kWN32 = 24, kWN64 = 40;

// ---------------------------------------------------------------------------------------
// Faddeeva function (Weideman); host and device, any floating type
// ---------------------------------------------------------------------------------------
template <typename T>
__host__ __device__ inline void faddeeva(T zr, T zi, const T* a, int N, T L, T& wr, T& wi) {
  // D = L - i z = (L + zi) - i zr;  1/D = conj(D)/|D|^2
  const T dr = L + zi, di = -zr;
  const T inv = T(1) / (dr * dr + di * di);
  const T ir = dr * inv, ii = -di * inv;
  // Z = (L + i z)/D = ((L - zi) + i zr)/D
  const T nr = L - zi, ni = zr;
  const T Zr = nr * ir - ni * ii, Zi = nr * ii + ni * ir;
  T pr = a[N - 1], pi = T(0);
  for (int j = N - 2; j >= 0; --j) {
    const T tr = pr * Zr - pi * Zi + a[j];
    pi = pr * Zi + pi * Zr;
    pr = tr;
  }
  // w = (1/D) (2 p / D + 1/sqrt(pi))
  const T qr = T(2) * (pr * ir - pi * ii) + T(0.56418958354775628695), qi = T(2) * (pr * ii + pi * ir);
  wr = ir * qr - ii * qi;
  wi = ir * qi + ii * qr;
}

static void weideman_coeffs(int N, double* a, double* L) {
  const int M = 2 * N, M2 = 2 * M;
  const double Lv = std::sqrt(N / std::sqrt(2.0));
  std::vector<double> f(M2, 0.0);
  for (int k = -M + 1; k <= M - 1; ++k) {
    const double th = k * M_PI / M, t = Lv * std::tan(th / 2.0);
    f[k + M] = std::exp(-t * t) * (Lv * Lv + t * t);
  }
  std::vector<double> g(M2);
  for (int j = 0; j < M2; ++j) g[j] = f[(j + M) % M2];  // the half-length rotation
  for (int m = 1; m <= N; ++m) {
    double re = 0.0;
    for (int j = 0; j < M2; ++j) re += g[j] * std::cos(2.0 * M_PI * (double)j * m / M2);
    a[m - 1] = re / M2;
  }
  *L = Lv;
}

struct WeidemanTables {
  double a32[kWMax], a64[kWMax];
  double L32, L64;
  WeidemanTables() {
    weideman_coeffs(kWN32, a32, &L32);
    weideman_coeffs(kWN64, a64, &L64);
  }
};

static const WeidemanTables& weideman() {
  static const WeidemanTables t;
  return t;
}

// ---------------------------------------------------------------------------------------
// decay-time terms
// ---------------------------------------------------------------------------------------
// V: float or double (one event), float2 (two events, packed FP32).
template <typename V>
struct TimeTerms {
  V P, Q, Tsh, Ts;
  V phi;  // N(t; 0, s)
};
template <typename V>
struct ScalarOf {
  using type = V;
};
template <>
struct ScalarOf<float2> {
  using type = float;
};

// Orders of the moment series (w_0 .. w_(2K+1)), and the largest
// z = max(|x|,|y|) G (max(t,0) + 6 s) at which the truncated
// series is used.  FP32: K = 4, z <= 0.5 (first omitted term of Q below 1e-8 of Q);
// FP64: K = 6, z <= 0.35 (below 1e-16 of Q).
template <typename T>
struct SeriesOrder {
  static constexpr int K = sizeof(T) == 4 ? 4 : 6;
  static constexpr double zmax = sizeof(T) == 4 ? 0.5 : 0.35;
};

// Per-theta constants of the decay-time terms in the path's precision, prepared on the host in
// FP64 from the rounded x, y, G and s.
template <typename T>
struct TimeCoef {
  static constexpr int K = SeriesOrder<T>::K;
  T G, x, y, s;
  T a[K + 1], b[K + 1];        // P, Q coefficients of w_2m (a_0 = 1, b_0 = 0)
  T ysh[K + 1], xs[K + 1];     // T_sh, T_s coefficients of w_(2m+1)
  // the order in use, K - 1 or K, and the observed time up to which it meets the truncation
  // criterion: K - 1 when that covers every event the dataset's time range admits
  int ku;
  T t_series;
  T t_gauss;                   // below it the FP32 Gaussian is subnormal
  T is2, is2h, ir2s;           // 1 / s^2, 1 / (2 s^2), 1 / (s sqrt 2): no event divides by them
  T k_phi;                     // 1 / (s sqrt(2 pi))
  T s2, Gs2, hG2s2;            // s^2, G s^2, G^2 s^2 / 2
  T nG2s2[2 * K + 1];          // n G^2 s^2
  T hx, hy, fx, fy;            // s^2 G x / 2, s^2 G y / 2, and twice these
  T Gx, Gy, qx, qy;            // G x, G y, 2 G^2 x, 2 G^2 y
  T Gx2, Gy2;                  // (G x)^2, (G y)^2
  // the Faddeeva path's: g = G (1 -+ y), g s^2 and g^2 s^2 / 2 of each; of g = G (1 - i x) the real part of
  // g^2 s^2 / 2 and the imaginary part of u
  T gp, gps2, hgp2s2, gm, gms2, hgm2s2, hgc2s2, ui;
};

#ifndef __CUDACC_RTC__
// t_hi: the upper limit of the observed time (events above it take the Faddeeva path where
// the order in use does not cover them, so it decides the speed, not the result).
template <typename T>
inline void fill_time_coef(TimeCoef<T>& c, double x64, double y64, double tau, double s64,
                           double t_hi = HUGE_VAL) {
  constexpr int K = TimeCoef<T>::K;
  c.G = (T)(1.0 / tau);
  c.x = (T)x64;
  c.y = (T)y64;
  c.s = (T)s64;
  const double x = (double)c.x, y = (double)c.y, G = (double)c.G, s = (double)c.s;
  const double zs = std::fmax(std::fabs(x), std::fabs(y)) * G;
  c.is2 = (T)(1.0 / (s * s));
  // FP32: t^2 times it stays finite up to the end of the range (the two-event exponential has no use for an
  // infinite argument); the Gaussian is 0 there all the same
  c.is2h = sizeof(T) == 4 ? (T)std::fmin(0.5 / (s * s), 3e38 / std::fmax(t_hi * t_hi, 1e-30)) : (T)(0.5 / (s * s));
  c.ir2s = (T)(0.70710678118654752440 / s);
  c.k_phi = (T)(0.39894228040143267794 / s);
  c.s2 = (T)(s * s);
  c.Gs2 = (T)(G * s * s);
  for (int n = 0; n <= 2 * K; ++n) c.nG2s2[n] = (T)(n * G * G * s * s);
  c.hG2s2 = (T)(0.5 * G * G * s * s);
  c.hx = (T)(0.5 * s * s * G * x);
  c.hy = (T)(0.5 * s * s * G * y);
  c.fx = (T)(s * s * G * x);
  c.fy = (T)(s * s * G * y);
  c.Gx = (T)(G * x);
  c.Gy = (T)(G * y);
  c.qx = (T)(2.0 * G * G * x);
  c.qy = (T)(2.0 * G * G * y);
  c.Gx2 = (T)(G * G * x * x);
  c.Gy2 = (T)(G * G * y * y);
  const double gp = G * (1.0 - y), gm = G * (1.0 + y);
  c.gp = (T)gp;
  c.gps2 = (T)(gp * s * s);
  c.hgp2s2 = (T)(0.5 * gp * gp * s * s);
  c.gm = (T)gm;
  c.gms2 = (T)(gm * s * s);
  c.hgm2s2 = (T)(0.5 * gm * gm * s * s);
  c.hgc2s2 = (T)(0.5 * G * G * s * s * (1.0 - x * x));
  c.ui = (T)(-G * x * s * 0.70710678118654752440);
  c.t_gauss = (T)(-s * std::sqrt(2.0 * 87.3));
  double fact = 1.0;  // (2m)!
  for (int m = 0; m <= K; ++m) {
    const double sg = (m & 1) ? -1.0 : 1.0;
    const double y2m = std::pow(y, 2 * m), x2m = std::pow(x, 2 * m);
    c.a[m] = (T)(0.5 * (y2m + sg * x2m) / fact);
    c.b[m] = (T)(0.5 * (y2m - sg * x2m) / fact);
    fact *= 2 * m + 1;
    c.ysh[m] = (T)(y2m * y / fact);
    c.xs[m] = (T)(sg * x2m * x / fact);
    fact *= 2 * m + 2;
  }
  c.b[0] = (T)0;
  // the first omitted term against the leading one is about z^(2k) 2 / (2k + 2)! at order k;
  // order K - 1 meets the bound that order K meets at SeriesOrder<T>::zmax up to zk1
  auto ratio = [](double z, int k) { return std::pow(z, 2.0 * k) * 2.0 / std::tgamma(2.0 * k + 3.0); };
  const double eps = ratio(SeriesOrder<T>::zmax, K);
  const double zk1 = std::pow(eps * std::tgamma(2.0 * (K - 1) + 3.0) / 2.0, 1.0 / (2.0 * (K - 1)));
  const double zdata = zs * (std::fmax(t_hi, 0.0) + 6.0 * s);
  c.ku = zdata < zk1 ? K - 1 : K;
  const double zlim = zdata < zk1 ? zk1 : SeriesOrder<T>::zmax;
  // z < zlim for max(t, 0) < zlim / zs - 6 s; never, where that is not positive
  const double tlim = zs > 0.0 ? zlim / zs - 6.0 * s : HUGE_VAL;
  c.t_series = (T)(tlim > 0.0 ? tlim : -HUGE_VAL);
}
#endif

// Products, sums and fused multiply-adds that the compiler neither fuses nor splits: the terms
// that enter log R are formed with them, so that an evaluation without the gradient (another
// instantiation of the kernels) returns the same NLL.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float2 mul_rn(float2 a, float2 b) { return pk::mul(a, b); }
__device__ __forceinline__ float2 sub_rn(float2 a, float2 b) { return pk::fma(b, pk::splat(-1.f), a); }
__device__ __forceinline__ float2 fma_rn(float2 a, float2 b, float2 c) { return pk::fma(a, b, c); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float2 add_rn(float2 a, float2 b) { return pk::add(a, b); }
// a scalar constant in every element of V
__device__ __forceinline__ float in(float, float c) { return c; }
__device__ __forceinline__ double in(double, double c) { return c; }
__device__ __forceinline__ float2 in(float2, float c) { return pk::splat(c); }

// R = |A|^2 P + |B|^2 Q + Re(A B*) T_sh + Im(A B*) T_s
template <typename V>
__device__ __forceinline__ V td_rate(const TimeTerms<V>& tt, V AA, V BB, V ABr, V ABi) {
  return fma_rn(ABi, tt.Ts, fma_rn(ABr, tt.Tsh, fma_rn(BB, tt.Q, mul_rn(AA, tt.P))));
}

// exp and erfcx / 2 of the path's precision: CUDA's for one FP32 event, the tables of fp64.cuh in FP64 and
// for two FP32 events.
template <typename V>
struct TdMath;
template <>
struct TdMath<float> {
  __device__ __forceinline__ float exp(float v) const { return expf(v); }
  // gauss erfcx(|u|) / 2
  __device__ __forceinline__ float gauss_herfcx(float gauss, float u) const {
    return mul_rn(mul_rn(0.5f, gauss), erfcxf(fabsf(u)));
  }
  __device__ __forceinline__ static bool nonneg(float u) { return u >= 0.f; }
  __device__ __forceinline__ static bool below(float t, float limit) { return t < limit; }
};
// Two events: exp from the hardware's 2^x of x log2(e) rounded once, the product's rounding error (an FMA gives
// it) applied as a factor; erfcx from its table in shared memory.  2^x is 0 below 2^-126: where a result
// there matters (the Gaussian of an event 13.2 resolutions below zero, the exponential 87 lifetimes above, whose
// rates are normal numbers) expf() takes over (exp_tail, for arguments below -87.3).
template <>
struct TdMath<float2> {
  const Fp32Tables& tab;
  __device__ __forceinline__ float2 exp(float2 v) const {
    const float2 np = mul_rn(v, pk::splat(-kLog2eHi));  // - v log2 e
    const float2 e = fma_rn(v, pk::splat(kLog2eLo), fma_rn(v, pk::splat(kLog2eHi), np));
    const float2 y = make_float2(pk::ex2(-np.x), pk::ex2(-np.y));
    return fma_rn(mul_rn(y, e), pk::splat(kLn2Hi), y);
  }
  __device__ __forceinline__ static void exp_tail(float2 v, float2& y) {
    if (v.x < -87.3f) y.x = expf(v.x);
    if (v.y < -87.3f) y.y = expf(v.y);
  }
  // gauss erfcx(|u|) / 2; where u <= -6 it is below 2^-52 of the exponential it is subtracted from
  // (conv_real) and is left out
  __device__ __forceinline__ float2 gauss_herfcx(float2 gauss, float2 u) const {
    const float2 a = make_float2(fminf(fabsf(u.x), (float)kErfcxMax), fminf(fabsf(u.y), (float)kErfcxMax));
    const float2 m = fma_rn(a, pk::splat((float)kErfcxStep), pk::splat(12582912.f));  // 1.5 2^23: the node in the low bits
    const float2 r = fma_rn(add_rn(m, pk::splat(-12582912.f)), pk::splat(-1.f / kErfcxStep), a);
    const int i0 = __float_as_int(m.x) & 0xff, i1 = __float_as_int(m.y) & 0xff;
    float2 p = make_float2(tab.herfcx[kErfcxDeg32][i0], tab.herfcx[kErfcxDeg32][i1]);
#pragma unroll
    for (int d = kErfcxDeg32 - 1; d >= 0; --d)
      p = fma_rn(p, r, make_float2(tab.herfcx[d][i0], tab.herfcx[d][i1]));
    float2 h = mul_rn(gauss, p);
    if (fabsf(u.x) > (float)kErfcxMax) h.x = u.x < 0.f ? 0.f : mul_rn(gauss.x, 0.5f * erfcxf(u.x));
    if (fabsf(u.y) > (float)kErfcxMax) h.y = u.y < 0.f ? 0.f : mul_rn(gauss.y, 0.5f * erfcxf(u.y));
    return h;
  }
};
template <>
struct TdMath<double> {
  const TimeTables& tab;
  __device__ __forceinline__ double exp(double v) const { return exp_tab(v, tab.exp); }
  // gauss erfcx(|u|) / 2; where u <= -6 it is below 2^-56 of the exponential it is subtracted from
  // (conv_real) and is left out
  __device__ __forceinline__ double gauss_herfcx(double gauss, double u) const {
    const int hu = __double2hiint(u), ha = hu & 0x7fffffff;
    if (ha < 0x40180000) return mul_rn(gauss, herfcx_tab(__hiloint2double(ha, __double2loint(u)), tab.erfcx));
    return hu < 0 ? 0.0 : mul_rn(gauss, 0.5 * erfcx(u));
  }
  // on the integer pipe (nonneg: false for -0, where both forms agree).  below: a double's high word with
  // the other bits of a negative one flipped is a signed integer that orders as the doubles do, whatever their signs
  // (t < 0 and the limit -inf, "never", among them); where the words are equal, t within 2^-20 of
  // the limit, the answer is no.
  __device__ __forceinline__ static bool nonneg(double u) { return __double2hiint(u) >= 0; }
  __device__ __forceinline__ static int ordered_high(double x) {
    const int h = __double2hiint(x);
    return h ^ ((h >> 31) & 0x7fffffff);
  }
  __device__ __forceinline__ static bool below(double t, double limit) { return ordered_high(t) < ordered_high(limit); }
};

// E(g) for real g (gauss = exp(-t^2/2s^2)): with h = gauss erfcx(|u|) / 2, u = (g s^2 - t) / (s sqrt 2),
// E = h for u >= 0 and exp(g^2 s^2 / 2 - g t) - h below, selected, so that a warp whose events
// lie on both sides evaluates erfcx once.  hg2s2 = g^2 s^2 / 2.
template <typename V, typename T>
__device__ __forceinline__ V conv_real(const TdMath<V>& F, T g, T gs2, T hg2s2, T ir2s, V t, V gauss) {
  const V z{};
  const V u = mul_rn(sub_rn(in(z, gs2), t), in(z, ir2s));
  const V h = F.gauss_herfcx(gauss, u);
  const V a = fma_rn(in(z, -g), t, in(z, hg2s2));
  V e = F.exp(a);
  if constexpr (sizeof(V) > sizeof(T)) {
    if (fminf(a.x, a.y) < -87.3f) F.exp_tail(a, e);
  }
  const V x = sub_rn(e, h);
  if constexpr (sizeof(V) > sizeof(T)) return make_float2(u.x >= 0.f ? h.x : x.x, u.y >= 0.f ? h.y : x.y);
  else return F.nonneg(u) ? h : x;
}

// The Faddeeva function as above, each operation rounded as written (see mul_rn).
template <typename T>
__device__ __forceinline__ void faddeeva_rn(T zr, T zi, const T* a, int N, T L, T& wr, T& wi) {
  const T dr = add_rn(L, zi), inv = T(1) / fma_rn(dr, dr, mul_rn(zr, zr));
  const T ir = mul_rn(dr, inv), ii = mul_rn(zr, inv);
  const T nr = sub_rn(L, zi);
  const T Zr = fma_rn(nr, ir, -mul_rn(zr, ii)), Zi = fma_rn(nr, ii, mul_rn(zr, ir));
  T pr = a[N - 1], pi = T(0);
  for (int j = N - 2; j >= 0; --j) {
    const T tr = fma_rn(pr, Zr, fma_rn(-pi, Zi, a[j]));
    pi = fma_rn(pr, Zi, mul_rn(pi, Zr));
    pr = tr;
  }
  const T qr = fma_rn(T(2), fma_rn(pr, ir, -mul_rn(pi, ii)), T(0.56418958354775628695));
  const T qi = mul_rn(T(2), fma_rn(pr, ii, mul_rn(pi, ir)));
  wr = fma_rn(ir, qr, -mul_rn(ii, qi));
  wi = fma_rn(ir, qi, mul_rn(ii, qr));
}

// The decay-time terms at the observed time t from the convolved exponentials (Faddeeva
// path, any mixing); gauss = exp(-t^2 / 2 s^2).  E of the complex g = G (1 - i x) by the same two forms as
// conv_real, u = (g s^2 - t) / (s sqrt 2).
template <typename T>
__device__ __forceinline__ void time_terms_direct(const TdMath<T>& F, const TimeCoef<T>& c, const T* wa, int wN, T wL,
                                                  T t, T gauss, TimeTerms<T>& R) {
  const T Ep = conv_real(F, c.gp, c.gps2, c.hgp2s2, c.ir2s, t, gauss);
  const T Em = conv_real(F, c.gm, c.gms2, c.hgm2s2, c.ir2s, t, gauss);
  const T v = sub_rn(t, c.Gs2), ur = mul_rn(-v, c.ir2s);
  const bool right = ur >= T(0);
  T wr, wi;  // w(i u), or w(-i u)
  faddeeva_rn<T>(right ? -c.ui : c.ui, right ? ur : -ur, wa, wN, wL, wr, wi);
  T Ecr = mul_rn(mul_rn(T(0.5), gauss), wr), Eci = mul_rn(mul_rn(T(0.5), gauss), wi);
  if (!right) {
    const T mag = F.exp(fma_rn(-c.G, t, c.hgc2s2)), ei = mul_rn(c.Gx, v);
    T sn, cs;
    if constexpr (sizeof(T) == 4) sincosf(ei, &sn, &cs);
    else sincos(ei, &sn, &cs);
    Ecr = fma_rn(mag, cs, -Ecr);
    Eci = fma_rn(mag, sn, -Eci);
  }
  const T Tch = mul_rn(T(0.5), add_rn(Ep, Em));
  R.P = mul_rn(T(0.5), add_rn(Tch, Ecr));
  R.Q = mul_rn(T(0.5), sub_rn(Tch, Ecr));
  R.Tsh = mul_rn(T(0.5), sub_rn(Ep, Em));
  R.Ts = Eci;
}

// The decay-time terms by the moment series of order KU (small mixing; see the top of this
// file).
template <typename V, typename T, int KU>
__device__ __forceinline__ void time_terms_series(const TdMath<V>& F, const TimeCoef<T>& c, V t, V gauss,
                                                  TimeTerms<V>& R) {
  constexpr int NW = 2 * KU + 2;
  const V z{};
  const V v = sub_rn(t, in(z, c.Gs2)), Gv = mul_rn(in(z, c.G), v);
  V w[NW];
  w[0] = conv_real(F, c.G, c.Gs2, c.hG2s2, c.ir2s, t, gauss);
  w[1] = mul_rn(in(z, c.G), fma_rn(v, w[0], mul_rn(in(z, c.s2), R.phi)));
#pragma unroll
  for (int n = 1; n < NW - 1; ++n) w[n + 1] = fma_rn(Gv, w[n], mul_rn(in(z, c.nG2s2[n]), w[n - 1]));
  R.P = w[0];
  R.Q = mul_rn(in(z, c.b[1]), w[2]);
  R.Tsh = mul_rn(in(z, c.ysh[0]), w[1]);
  R.Ts = mul_rn(in(z, c.xs[0]), w[1]);
#pragma unroll
  for (int m = 1; m <= KU; ++m) {
    R.P = fma_rn(in(z, c.a[m]), w[2 * m], R.P);
    if (m > 1) R.Q = fma_rn(in(z, c.b[m]), w[2 * m], R.Q);
    R.Tsh = fma_rn(in(z, c.ysh[m]), w[2 * m + 1], R.Tsh);
    R.Ts = fma_rn(in(z, c.xs[m]), w[2 * m + 1], R.Ts);
  }
}

// The decay-time terms at the observed time t: the moment series of the
// order in use where z = max(|x|, |y|) G (max(t, 0) + 6 s) is below its limit (t < c.t_series),
// else the Faddeeva path.
template <typename T>
__device__ __forceinline__ void time_terms_g(const TdMath<T>& F, const TimeCoef<T>& c, const T* wa, int wN, T wL, T t,
                                             TimeTerms<T>& R) {
  const T gauss = F.exp(mul_rn(mul_rn(-t, t), c.is2h));
  R.phi = mul_rn(c.k_phi, gauss);
  if (F.below(t, c.t_series)) {
    // the same order for every event of a launch (a uniform branch)
    if (c.ku == TimeCoef<T>::K) time_terms_series<T, T, TimeCoef<T>::K>(F, c, t, gauss, R);
    else time_terms_series<T, T, TimeCoef<T>::K - 1>(F, c, t, gauss, R);
  } else {
    time_terms_direct<T>(F, c, wa, wN, wL, t, gauss, R);
  }
}

// The same for two events, packed; an event above the series' limit goes through the scalar code.
__device__ __forceinline__ void time_terms_pair(const TdMath<float2>& F, const TimeCoef<float>& c, const float* wa,
                                                int wN, float wL, float2 t, TimeTerms<float2>& R) {
  const float2 q = mul_rn(mul_rn(mul_rn(t, pk::splat(-1.f)), t), pk::splat(c.is2h));
  float2 gauss = F.exp(q);
  if (fminf(t.x, t.y) < c.t_gauss) F.exp_tail(q, gauss);
  R.phi = mul_rn(pk::splat(c.k_phi), gauss);
  if (c.ku == TimeCoef<float>::K) time_terms_series<float2, float, TimeCoef<float>::K>(F, c, t, gauss, R);
  else time_terms_series<float2, float, TimeCoef<float>::K - 1>(F, c, t, gauss, R);
  if (!(t.x < c.t_series && t.y < c.t_series)) {
#pragma unroll 1
    for (int e = 0; e < 2; ++e) {
      const float te = e ? t.y : t.x;
      if (te < c.t_series) continue;
      TimeTerms<float> S;
      time_terms_direct<float>(TdMath<float>{}, c, wa, wN, wL, te, expf(mul_rn(mul_rn(-te, te), c.is2h)), S);
      (e ? R.P.y : R.P.x) = S.P;
      (e ? R.Q.y : R.Q.x) = S.Q;
      (e ? R.Tsh.y : R.Tsh.x) = S.Tsh;
      (e ? R.Ts.y : R.Ts.x) = S.Ts;
    }
  }
}

// Adds one event's lanes X / R, Y / R, Z / R and the d^2 / dt^2 bracket / R (see the top of this
// file) to lt; AA = |A|^2, BB = |B|^2, (ABr, ABi) = A conj(B).
template <typename V, typename T>
__device__ __forceinline__ void time_lanes(const TimeCoef<T>& c, V t, const TimeTerms<V>& tt, V AA, V BB, V ABr, V ABi,
                                           V invR, V (&lt)[4]) {
  const V z{};
  auto K = [&](T x) { return in(z, x); };
  const V v = sub_rn(t, K(c.Gs2));
  const V Tch = add_rn(tt.P, tt.Q), Tc = sub_rn(tt.P, tt.Q);
  const V ysh = mul_rn(K(c.hy), tt.Tsh), xs = mul_rn(K(c.hx), tt.Ts);
  const V CP = fma_rn(v, tt.P, fma_rn(K(c.s2), tt.phi, sub_rn(ysh, xs))), CQ = fma_rn(v, tt.Q, add_rn(ysh, xs));
  const V Csh = fma_rn(v, tt.Tsh, mul_rn(K(c.fy), Tch)), Cs = fma_rn(v, tt.Ts, mul_rn(K(c.fx), Tc));
  const V hp = mul_rn(K(T(0.5)), add_rn(AA, BB)), hm = mul_rn(K(T(0.5)), sub_rn(BB, AA));
  lt[0] = fma_rn(fma_rn(hm, Cs, mul_rn(ABi, sub_rn(CP, CQ))), invR, lt[0]);
  lt[1] = fma_rn(fma_rn(hp, Csh, mul_rn(ABr, add_rn(CP, CQ))), invR, lt[1]);
  lt[2] = fma_rn(fma_rn(AA, CP, fma_rn(BB, CQ, fma_rn(ABr, Csh, mul_rn(ABi, Cs)))), invR, lt[2]);
  // E_y, E_x, R_y and R_x each times its factor: G^2 (y^2 R_y - x^2 R_x - 2 (y E_y + x E_x))
  const V Ey = fma_rn(hp, tt.Tsh, mul_rn(ABr, Tch)), Ex = fma_rn(hm, tt.Ts, mul_rn(ABi, Tc));
  const V Ry = fma_rn(hp, Tch, mul_rn(ABr, tt.Tsh)), mRx = fma_rn(hm, Tc, mul_rn(K(T(-1)), mul_rn(ABi, tt.Ts)));
  const V b = fma_rn(fma_rn(t, K(-c.is2), K(-c.G)), AA, fma_rn(K(c.Gy), ABr, mul_rn(K(c.Gx), ABi)));
  const V q = fma_rn(tt.phi, b,
                     fma_rn(K(c.Gy2), Ry, fma_rn(K(c.Gx2), mRx, fma_rn(K(-c.qy), Ey, mul_rn(K(-c.qx), Ex)))));
  lt[3] = fma_rn(q, invR, lt[3]);
}

// sum_i (dR_i / dp_j) / R_i of j = x, y, tau, sigma_t from the lane sums of n events (FP64).
__device__ __forceinline__ double time_gradient(int j, double G, double x, double y, double s, const double* lanes,
                                                double n) {
  if (j == 0) return G * lanes[0];
  if (j == 1) return G * lanes[1];
  if (j == 2) return G * G * (lanes[2] - y * lanes[1] - x * lanes[0]);  // -G (G d / dG)
  return s * (G * G * n + lanes[3]);
}

}  // namespace goo
