// dalitz.cuh -- device code shared by the amplitude-model kernels (dalitz.cu) and the
// toy-MC server (serve.cu): lineshape constants, the Breit-Wigner amplitude of one
// resonance, and the loads of the cached amplitudes of one event.  The formulas are stated
// at the top of dalitz.cu.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace goo {

constexpr int kMaxAmp = 16;

template <typename T>
struct BwConstT {
  int spin, pair;  // pair 0: (12)+3, 1: (13)+2, 2: (23)+1
  T m0sq, m0w;     // m0^2, m0 * Gamma0
  T inv_q0sq;      // 1 / q0^2
  T r2, rp2;       // resonance and parent barrier radii squared
  T thrP, thrM;    // (mA + mB)^2, (mA - mB)^2
  T pthrP, pthrM;  // (M + mC)^2, (M - mC)^2
  T zconst;        // (mA^2 - mB^2)(M^2 - mC^2)
  T inv4M2;        // 1 / (4 M^2)
  T Fz0;           // 1 + z0 (L=1) or 9 + 3 z0 + z0^2 (L=2)
  T m0;            // m0
};
using BwConst = BwConstT<double>;

struct DalitzDev {
  int nbw;              // number of Breit-Wigner amplitudes (cached)
  double sumsq;         // M^2 + m1^2 + m2^2 + m3^2  (s23 = sumsq - s12 - s13)
  BwConstT<double> bw[kMaxAmp];
  BwConstT<float> bwf[kMaxAmp];  // the same constants rounded to float (FP32 path)
};

// ---------------------------------------------------------------------------------------
// amplitude of one Breit-Wigner resonance at (s12, s13, s23), in precision T
// ---------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void bw_amp(const BwConstT<T>& b, T s12, T s13, T s23, T& re, T& im) {
  const int L = b.spin;
  T s, sac, sbc;
  if (b.pair == 0) {
    s = s12;
    sac = s13;
    sbc = s23;
  } else if (b.pair == 1) {
    s = s13;
    sac = s12;
    sbc = s23;
  } else {
    s = s23;
    sac = s12;
    sbc = s13;
  }
  const T lam1 = (s - T(b.thrP)) * (s - T(b.thrM));
  T q2 = lam1 / (T(4) * s);
  q2 = q2 > T(0) ? q2 : T(0);
  const T z = T(b.r2) * q2;
  const T t = q2 * T(b.inv_q0sq);
  const T st = sqrt(t);
  T ratio2, pw;
  if (L == 0) {
    ratio2 = T(1);
    pw = st;
  } else if (L == 1) {
    ratio2 = T(b.Fz0) / (T(1) + z);
    pw = t * st;
  } else {
    ratio2 = T(b.Fz0) / (T(9) + T(3) * z + z * z);
    pw = t * t * st;
  }
  const T rs = T(1) / sqrt(s);
  const T m0 = b.m0;
  const T di = T(b.m0w) * pw * m0 * rs * ratio2;  // m0 Gamma(s)
  const T dr = T(b.m0sq) - s;
  const T inv = T(1) / (dr * dr + di * di);
  const T lam2 = (s - T(b.pthrP)) * (s - T(b.pthrM));
  T zp = T(b.rp2) * lam2 * T(b.inv4M2);
  zp = zp > T(0) ? zp : T(0);
  T parent, spinf;
  if (L == 0) {
    parent = T(1);
    spinf = T(1);
  } else if (L == 1) {
    parent = T(1) / sqrt(T(1) + zp);
    spinf = sac - sbc - T(b.zconst) / s;
  } else {
    parent = T(3) / sqrt(T(9) + T(3) * zp + zp * zp);
    const T z1 = sac - sbc - T(b.zconst) / s;
    spinf = z1 * z1 - lam1 * lam2 / (T(3) * s * s);
  }
  const T scale = sqrt(ratio2) * parent * spinf * inv;
  re = dr * scale;
  im = di * scale;
}

// Loads the nbw cached amplitudes of event i (compile-time bound KB, runtime nbw).
template <int KB>
__device__ __forceinline__ void load_amps(const float4* __restrict__ cache, int64_t n, int64_t i, int nbw,
                                          float (&ar)[KB + 1], float (&ai)[KB + 1]) {
#pragma unroll
  for (int p = 0; p < (KB + 1) / 2; ++p) {
    if (2 * p < nbw) {
      const float4 v = __ldg(cache + (int64_t)p * n + i);
      ar[2 * p] = v.x;
      ai[2 * p] = v.y;
      if (2 * p + 1 < KB) {
        ar[2 * p + 1] = v.z;
        ai[2 * p + 1] = v.w;
      }
    } else {
      ar[2 * p] = ai[2 * p] = 0.f;
      if (2 * p + 1 < KB) ar[2 * p + 1] = ai[2 * p + 1] = 0.f;
    }
  }
}

template <int KB>
__device__ __forceinline__ void load_amps(const double2* __restrict__ cache, int64_t n, int64_t i, int nbw,
                                          double (&ar)[KB + 1], double (&ai)[KB + 1]) {
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    if (k < nbw) {
      const double2 v = cache[(int64_t)k * n + i];
      ar[k] = v.x;
      ai[k] = v.y;
    } else {
      ar[k] = ai[k] = 0.0;
    }
  }
}

// One event of a coherent sum in packed FP32 form.  With a_k = (Re A_k, Im A_k) of the KB resonance slots
// held as a register pair, cre_k = (Re c_k, Re c_k), cim_k = (Im c_k, Im c_k) and the constant amplitude 1 in
// slot KB:
//   P = sum_k Re c_k a_k,  Q = sum_k Im c_k a_k,  S = (P.x - Q.y) + i (P.y + Q.x),
// and the gradient lanes A_k conj(S) / |S|^2 = (t_r + i t_i) A_k are accumulated as
//   G1_k += t_r a_k,  G2_k += t_i a_k   (Re = G1.x - G2.y, Im = G1.y + G2.x at the end),
// so each resonance costs two packed fma for S and two for the gradient, the constant two additions.
template <int KB, bool GRAD>
__device__ __forceinline__ void coh_event_pk(const float2 (&cre)[KB + 1], const float2 (&cim)[KB + 1],
                                             const float2 (&a)[KB], Kahan& lf, float2 (&G1)[KB + 1],
                                             float2 (&G2)[KB + 1], unsigned& bad) {
  float2 P = make_float2(cre[KB].x, 0.f), Q = make_float2(cim[KB].x, 0.f);
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    P = pk::fma(cre[k], a[k], P);
    Q = pk::fma(cim[k], a[k], Q);
  }
  const float sr = P.x - Q.y, si = P.y + Q.x;
  const float s2 = fmaf(sr, sr, si * si);
  if (s2 > 0.f) {
    lf.add(pk::kLn2 * pk::lg2(s2));
    if constexpr (GRAD) {
      const float inv = pk::rcp(s2);
      const float tr = sr * inv, ti = -si * inv;  // conj(S) / |S|^2
      const float2 tr2 = pk::splat(tr), ti2 = pk::splat(ti);
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        G1[k] = pk::fma(tr2, a[k], G1[k]);
        G2[k] = pk::fma(ti2, a[k], G2[k]);
      }
      G1[KB].x += tr;
      G2[KB].x += ti;
    }
  } else {
    bad++;
  }
}

}  // namespace goo
