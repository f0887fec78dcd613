// lineshape.cuh -- Breit-Wigner amplitudes of the three-body models at one Dalitz point, arranged so
// that what depends on the pair and the spin alone is computed once per point, not once per
// resonance (formulas at the top of dalitz.cu).
//
// For a resonance k of spin L in a pair with invariant mass squared s,
//   m0 Gamma(s) = c1_k g,   g = q^(2L+1) / (sqrt(s) F_L(z)),     c1_k = m0^2 Gamma0 F_L(z0) / q0^(2L+1),
//   A_k = c2_k h (dr + i di) / (dr^2 + di^2),  dr = m0^2 - s, di = c1_k g,   c2_k = sqrt(F_L(z0)),
//   h = Z_L / sqrt(F_L(z) F_L(z_p)),
// with F_0 = 1, F_1(z) = 1 + z, F_2(z) = 9 + 3z + z^2 (the squared barriers are 1/F_1 and 9/F_2),
// z = r^2 q^2, z_p = r_par^2 p*^2 and Z_L the spin factor.  g and h are shared by every resonance of
// the pair and spin: at most nine of them per point, and ten operations and one reciprocal per resonance
// instead of some 150 instructions with six divisions and four square roots.
//
// The FP32 code works on two points at a time (packed .f32x2 arithmetic); reciprocals and
// reciprocal square roots are the hardware approximations sharpened by one Newton step (FP64:
// one third-order step).
#pragma once

#include "common.cuh"
#include "dalitz.cuh"
#include "fp64.cuh"

namespace goo {

template <typename T>
struct LsTables {
  T sum_hi, sum_lo;  // M^2 + m1^2 + m2^2 + m3^2 (lo: the rounding error of hi, FP32 only)
  T r2, zpk;         // r_res^2, r_par^2 / (4 M^2)
  struct Pair {
    T thrP, thrM, pthrP, pthrM, zconst;  // (mA +- mB)^2, (M +- mC)^2, (mA^2 - mB^2)(M^2 - mC^2)
  } pair[3];
  struct Res {
    T m0sq, c1, c2;
    int group;  // 3 pair + L
  } res[kMaxAmp];
  int nbw, groups;  // groups: bit g set when some resonance is of group g
};

// --- arithmetic on one double or a pair of floats ---------------------------------------
namespace lsv {
__device__ __forceinline__ double splat(double, double x) { return x; }
__device__ __forceinline__ float2 splat(float2, float x) { return pk::splat(x); }
__device__ __forceinline__ double mul(double a, double b) { return a * b; }
__device__ __forceinline__ float2 mul(float2 a, float2 b) { return pk::mul(a, b); }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ float2 add(float2 a, float2 b) { return pk::add(a, b); }
__device__ __forceinline__ double sub(double a, double b) { return a - b; }
// a - b as an FMA by -1 and a negation as a product by -1 (exact): one packed instruction each
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return pk::fma(b, pk::splat(-1.f), a); }
__device__ __forceinline__ double fma(double a, double b, double c) { return ::fma(a, b, c); }
__device__ __forceinline__ float2 fma(float2 a, float2 b, float2 c) { return pk::fma(a, b, c); }
__device__ __forceinline__ float2 neg(float2 a) { return pk::mul(a, pk::splat(-1.f)); }
__device__ __forceinline__ double neg(double a) { return -a; }
__device__ __forceinline__ float2 floor_at(float2 a, float lo) { return make_float2(fmaxf(a.x, lo), fmaxf(a.y, lo)); }
// lo >= 0: the sign and the magnitude are compared as integers
__device__ __forceinline__ double floor_at(double a, double lo) {
  return __double_as_longlong(a) > __double_as_longlong(lo) ? a : lo;
}
// 1 / x, x > 0
__device__ __forceinline__ double rcp(double x) { return rcp64(x); }
__device__ __forceinline__ float2 rcp(float2 x) {
  const float2 y = pk::rcp(x);
  return fma(y, fma(x, neg(y), pk::splat(1.f)), y);
}
// 1 / sqrt(x), x > 0
__device__ __forceinline__ double rsqrt(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = ::fma(-(x * y), y, 1.0);  // y (1 + e/2 + 3 e^2 / 8), the binomial series of (1 - e)^(-1/2)
  return ::fma(y * e, ::fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ float rsqrt1(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float2 rsqrt(float2 x) {
  const float2 y = make_float2(rsqrt1(x.x), rsqrt1(x.y));
  const float2 e = fma(mul(x, y), y, pk::splat(-1.f));  // x y^2 - 1
  return fma(mul(pk::splat(-0.5f), y), e, y);
}
// M^2 + sum m_i^2 - a - b to full precision: in FP32 from the exact differences (a < sum, b < sum - a)
__device__ __forceinline__ double third(const LsTables<double>& t, double a, double b) { return t.sum_hi - a - b; }
__device__ __forceinline__ float2 third(const LsTables<float>& t, float2 a, float2 b) {
  const float2 h = pk::splat(t.sum_hi);
  const float2 d = sub(h, a), ed = sub(sub(h, d), a);
  const float2 c = sub(d, b), ec = sub(sub(d, c), b);
  return add(c, add(add(ed, ec), pk::splat(t.sum_lo)));
}
}  // namespace lsv

// Smallest q^2 used (q^2 <= 0 at and beyond the pair's threshold): its root stays normal.
template <typename T>
__device__ __forceinline__ T ls_q2_floor() {
  return sizeof(T) == 4 ? T(1e-30) : T(1e-200);
}

// The shared factors of the model's groups at (a, b) = (s12, s13) into the thread's column of
// shared memory: s of pair p at sc[p * stride], g and h of group j at gc[j * stride], hc[j * stride].
template <typename T, typename V>
__device__ __forceinline__ void ls_groups(const LsTables<T>& t, V a, V b, V* sc, V* gc, V* hc, int stride) {
  using namespace lsv;
  const V c = third(t, a, b);
  const V one = splat(V{}, T(1));
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const int used = (t.groups >> (3 * p)) & 7;
    if (!used) continue;
    const V s = p == 0 ? a : (p == 1 ? b : c);
    const V sac = p == 0 ? b : a, sbc = p == 2 ? b : c;  // (12): s13, s23; (13): s12, s23; (23): s12, s13
    const typename LsTables<T>::Pair& P = t.pair[p];
    const V rs = rsqrt(s), is = rcp(s);
    const V lam1 = mul(sub(s, splat(V{}, P.thrP)), sub(s, splat(V{}, P.thrM)));
    const V q2 = floor_at(mul(mul(lam1, is), splat(V{}, T(0.25))), ls_q2_floor<T>());
    const V qrs = mul(mul(q2, rsqrt(q2)), rs);  // q / sqrt(s)
    sc[p * stride] = s;
    if (used & 1) {
      gc[3 * p * stride] = qrs;
      hc[3 * p * stride] = one;
    }
    if (!(used & 6)) continue;
    const V z = mul(splat(V{}, t.r2), q2);
    const V lam2 = mul(sub(s, splat(V{}, P.pthrP)), sub(s, splat(V{}, P.pthrM)));
    const V zp = floor_at(mul(splat(V{}, t.zpk), lam2), T(0));
    const V z1 = sub(sub(sac, sbc), mul(splat(V{}, P.zconst), is));
    const V q3rs = mul(qrs, q2);
    if (used & 2) {
      const V F = add(one, z);
      gc[(3 * p + 1) * stride] = mul(q3rs, rcp(F));
      hc[(3 * p + 1) * stride] = mul(z1, rsqrt(mul(F, add(one, zp))));
    }
    if (used & 4) {
      const V three = splat(V{}, T(3)), nine = splat(V{}, T(9));
      const V F = fma(z, add(z, three), nine), Fp = fma(zp, add(zp, three), nine);
      const V Z2 = fma(z1, z1, mul(mul(lam1, lam2), mul(mul(is, is), splat(V{}, T(-1.0 / 3.0)))));
      gc[(3 * p + 2) * stride] = mul(mul(q3rs, q2), rcp(F));
      // the parent's barrier at z_p = 0 is 1: sqrt(9 / F_2)
      hc[(3 * p + 2) * stride] = mul(mul(splat(V{}, T(3)), Z2), rsqrt(mul(F, Fp)));
    }
  }
}

// Amplitude k, A = h / D with a real numerator h, from the shared factors: di of D = dr - i di,
template <typename T, typename V>
__device__ __forceinline__ V ls_width(const LsTables<T>& t, int k, const V* gc, int stride) {
  return lsv::mul(lsv::splat(V{}, t.res[k].c1), gc[t.res[k].group * stride]);
}
// 1 / D = gr + i gi, and di,
template <typename T, typename V>
__device__ __forceinline__ void ls_propagator(const LsTables<T>& t, int k, const V* sc, const V* gc, int stride, V& gr,
                                              V& gi, V& di) {
  using namespace lsv;
  const typename LsTables<T>::Res& R = t.res[k];
  const V dr = sub(splat(V{}, R.m0sq), sc[R.group / 3 * stride]);
  di = ls_width<T, V>(t, k, gc, stride);
  const V inv = rcp(fma(dr, dr, mul(di, di)));
  gr = mul(dr, inv);
  gi = mul(di, inv);
}
// and h.
template <typename T, typename V>
__device__ __forceinline__ V ls_numerator(const LsTables<T>& t, int k, const V* hc, int stride) {
  using namespace lsv;
  const typename LsTables<T>::Res& R = t.res[k];
  return mul(splat(V{}, R.c2), hc[R.group * stride]);
}
template <typename T, typename V>
__device__ __forceinline__ void ls_amp(const LsTables<T>& t, int k, const V* sc, const V* gc, const V* hc, int stride,
                                       V& re, V& im) {
  using namespace lsv;
  V gr, gi, di;
  ls_propagator<T, V>(t, k, sc, gc, stride, gr, gi, di);
  const V h = ls_numerator<T, V>(t, k, hc, stride);
  re = mul(gr, h);
  im = mul(gi, h);
}

// Threads per block of the kernels that keep the shared factors in shared memory: 21 values per
// thread (packed pairs or doubles, 168 bytes).
constexpr int kLsBlock = 128;
constexpr int kLsCols = 21;

}  // namespace goo
