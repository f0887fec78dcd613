// td4.cu -- the time-dependent four-body amplitude model: amplitude cache, MC Gram matrix,
// and the NLL + adjoint gradient with mixing and a Gaussian decay-time resolution.
//
// Paper: a time-dependent amplitude analysis of four-body decays for a mixing measurement
// is among GooFit's amplitude PDFs (Sec. 5); phase-space MC samples give the normalisation
// (Sec. 5); partial results are cached in structure-of-arrays form (Sec. 4).  The paper
// prints no formulas; the model (fixed by the oracle) is:
//   observables m12, m34, c12 = cos th12, c34 = cos th34, phi, t;
//   a_k = F(m12) F(m34) W_k(c12, c34, phi),  F = BW(m^2) (q/q0)^L B_L(r q)/B_L(r q0),
//   BW(s) = 1/(m0^2 - s - i m0 G(m)),  G(m) = G0 (q/q0)^(2L+1) (m0/m) (B_L(rq)/B_L(rq0))^2;
//   A = sum_k c_k a_k (free), B = sum_k b_k a_k (fixed);
//   R = (|A|^2+|B|^2)/2 T_ch + (|A|^2-|B|^2)/2 T_c + Re(AB*) T_sh + Im(AB*) T_s,
//   T_ch, T_sh = (E(G(1-y)) +- E(G(1+y)))/2,  T_c + i T_s = E(G(1 - i x)),  G = 1/tau,
//   E(g; t, s) = e^{-g t'} (t' >= 0) convolved with N(0, s):
//     Re u >= 0:  E = 1/2 exp(-t^2/2s^2) w(i u),  u = (g s^2 - t)/(s sqrt 2)
//     Re u <  0:  E = exp(g^2 s^2/2 - g t) - 1/2 exp(-t^2/2s^2) w(-i u);
//   N = <|A|^2+|B|^2>/2 I_ch + <|A|^2-|B|^2>/2 I_c + Re<AB*> I_sh + Im<AB*> I_s over the MC
//   (Gram matrix <a_k a_l*>), I_ch = tau/(1-y^2), I_sh = y tau/(1-y^2), I_c = tau/(1+x^2),
//   I_s = x tau/(1+x^2);  NLL = -sum log R + n log N.
// The Faddeeva function w(z), Im z >= 0, is Weideman's rational approximation (J. A. C.
// Weideman, SIAM J. Numer. Anal. 31 (1994) 1497):
//   w(z) = 2 p(Z)/(L - iz)^2 + (1/sqrt pi)/(L - iz),  Z = (L + iz)/(L - iz),  L = sqrt(N/sqrt 2),
// p a polynomial of degree N-1 whose coefficients come from a discrete Fourier transform of
// exp(-t^2)(L^2 + t^2) at t = L tan(theta/2) (computed here on the host in FP64); N = 24 in
// the FP32 path and 40 in the FP64 path.  The real-argument terms use erfcx.
//
// Gradient lanes per event: log R; Re, Im of a_k V / R with
// V = (T_ch + T_c) A* + (T_sh - i T_s) B* (dR/dRe c_k = Re(a_k V), dR/dIm c_k = -Im(a_k V));
// and the four decay-time lanes of timeterms.cuh.  The last block forms the NLL and its gradient in FP64.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "gram.cuh"
#include "model.cuh"
#include "timeterms.cuh"

namespace goo {

constexpr int kTdMaxAmp = 16;

struct Td4Amp {
  int ang, L1, L2, pad;
  double m0a, g0a, q0a, b0a;  // resonance in the 12 pair: m0, width, q(m0), B_L(r q(m0))
  double m0b, g0b, q0b, b0b;  // resonance in the 34 pair
};

struct Td4Dev {
  int K, pad;
  double m1, m2, m3, m4, r;
  Td4Amp amp[kTdMaxAmp];
  double br[kTdMaxAmp], bi[kTdMaxAmp];  // the model's constant coefficients of B = sum b_k a_k
};

template <typename T>
struct Td4Args {
  T cr[kTdMaxAmp], ci[kTdMaxAmp], br[kTdMaxAmp], bi[kTdMaxAmp];
  T G, x, y, s;  // 1/tau, mixing, resolution in the path's precision
  TimeCoef<T> tc;  // the same with the moment-series coefficients (timeterms.cuh)
  T wa[kWMax];   // Weideman coefficients (constant term first)
  T wL;
  int wN, K, n_params, planes;
  // terms 2k, 2k + 1: the coefficient parameters of amplitude k; 2 kTdMaxAmp + j: the time parameters
  GradMap<2 * kTdMaxAmp + 4> map;
  int64_t n_total;  // events of the dataset (cache plane length)
  int has_b;        // FP64: the cache holds B in plane K
  // the normalisation at theta, formed on the host in FP64 from the cached Gram matrix
  // (td4_norm_terms): N, log N, (dN / d Re c_k) / N, (dN / d Im c_k) / N and (dN / dx) / N,
  // (dN / dy) / N, (tau dN / d tau) / N
  double nrm_N, nrm_logN, nrm_ur[kTdMaxAmp], nrm_ui[kTdMaxAmp], nrm_dt[3];
};


// ---------------------------------------------------------------------------------------
// amplitude cache
// ---------------------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T td_barrier(int L, T z) {
  if (L == 0) return T(1);
  if (L == 1) return sqrt(T(1) / (T(1) + z));
  return sqrt(T(9) / (T(9) + T(3) * z + z * z));
}

template <typename T>
__device__ __forceinline__ void td_lineshape(T m, T m0, T g0, T q0, T b0, int L, T ma, T mb, T r, T& fr, T& fi) {
  const T m2 = m * m;
  const T lam = (m2 - (ma + mb) * (ma + mb)) * (m2 - (ma - mb) * (ma - mb));
  const T q = sqrt(lam > T(0) ? lam : T(0)) / (T(2) * m);
  const T ratio = td_barrier<T>(L, (r * q) * (r * q)) / b0;
  const T qq = q / q0;
  T qL = T(1);
  for (int l = 0; l < L; ++l) qL *= qq;
  const T width = g0 * qL * qL * qq * (m0 / m) * ratio * ratio;
  const T dr = m0 * m0 - m2, di = m0 * width;  // BW = 1/(dr - i di) = (dr + i di)/|.|^2
  const T inv = T(1) / (dr * dr + di * di);
  const T scale = qL * ratio * inv;
  fr = dr * scale;
  fi = di * scale;
}

template <typename T>
__device__ __forceinline__ void td_angular(int ang, T c12, T c34, T phi, T& wr, T& wi) {
  const T s12 = sqrt(fmax(T(1) - c12 * c12, T(0))), s34 = sqrt(fmax(T(1) - c34 * c34, T(0)));
  const T p2 = T(0.5) * (T(3) * c12 * c12 - T(1));
  wi = T(0);
  switch (ang) {
    case GOO_ANG_SS: wr = T(1); break;
    case GOO_ANG_VS0: wr = c12; break;
    case GOO_ANG_SV0: wr = c34; break;
    case GOO_ANG_VV0: wr = c12 * c34; break;
    case GOO_ANG_VVPAR: wr = s12 * s34 * cos(phi); break;
    case GOO_ANG_VVPERP: wr = T(0); wi = s12 * s34 * sin(phi); break;
    case GOO_ANG_TS0: wr = p2; break;
    default: wr = p2 * c34; break;  // GOO_ANG_TV0
  }
}

template <typename T>
struct Td4Cols {
  const T* c[5];  // m12, m34, c12, c34, phi
};

// B += b a, one order of operations wherever B is formed
__device__ __forceinline__ void td4_add_b(double br, double bi, double2 a, double& Br, double& Bi) {
  Br = fma_rn(br, a.x, fma_rn(-bi, a.y, Br));
  Bi = fma_rn(br, a.y, fma_rn(bi, a.x, Bi));
}

// Cache layout as for the three-body model: FP32 ceil(K/2) planes of float4 (re_k, im_k,
// re_k+1, im_k+1), FP64 K planes of double2; plane p of an n-event dataset at p * n.  FP64, with_b: B = sum b_k a_k,
// whose coefficients are the model's constants, in plane K (16 bytes more an event where B costs the
// evaluation 4 K slots of the FP64 pipe).
template <typename T>
__global__ void td4_cache_kernel(const Td4Dev* __restrict__ tdp, Td4Cols<T> cols, int64_t n, void* cache_v, bool with_b) {
  __shared__ Td4Dev td;
  for (int i = threadIdx.x; i < (int)(sizeof(Td4Dev) / 4); i += blockDim.x) ((int*)&td)[i] = ((const int*)tdp)[i];
  __syncthreads();
  const int K = td.K;
  const T r = (T)td.r;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const T m12 = cols.c[0][i], m34 = cols.c[1][i], c12 = cols.c[2][i], c34 = cols.c[3][i], phi = cols.c[4][i];
    double Br = 0.0, Bi = 0.0;
    for (int k = 0; k < K; ++k) {
      const Td4Amp& A = td.amp[k];
      T f1r, f1i, f2r, f2i, wr, wi;
      td_lineshape<T>(m12, (T)A.m0a, (T)A.g0a, (T)A.q0a, (T)A.b0a, A.L1, (T)td.m1, (T)td.m2, r, f1r, f1i);
      td_lineshape<T>(m34, (T)A.m0b, (T)A.g0b, (T)A.q0b, (T)A.b0b, A.L2, (T)td.m3, (T)td.m4, r, f2r, f2i);
      td_angular<T>(A.ang, c12, c34, phi, wr, wi);
      const T fr = f1r * f2r - f1i * f2i, fi = f1r * f2i + f1i * f2r;
      const T ar = fr * wr - fi * wi, ai = fr * wi + fi * wr;
      if constexpr (sizeof(T) == 4) {
        float* plane = (float*)((float4*)cache_v + (int64_t)(k / 2) * n + i);
        plane[2 * (k & 1)] = ar;
        plane[2 * (k & 1) + 1] = ai;
      } else {
        ((double2*)cache_v)[(int64_t)k * n + i] = make_double2(ar, ai);
        td4_add_b(td.br[k], td.bi[k], make_double2(ar, ai), Br, Bi);
      }
    }
    if (sizeof(T) == 8 && with_b) ((double2*)cache_v)[(int64_t)K * n + i] = make_double2(Br, Bi);
    if constexpr (sizeof(T) == 4) {
      if (K & 1) {  // zero the unused half of the last plane
        float* plane = (float*)((float4*)cache_v + (int64_t)(K / 2) * n + i);
        plane[2] = plane[3] = 0.f;
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// NLL kernels
// ---------------------------------------------------------------------------------------
template <int KB, bool GRAD>
struct TdLanes {
  static constexpr int NS = GRAD ? 1 + 2 * KB + 4 : 1;
};

template <typename T, int KB>
struct TdAcc {
  ddf lf;  // the thread's sum of log R
  T lre[KB], lim[KB], lt[4];
  unsigned bad = 0;
};

// The FP32 sums of one event.  The amplitudes come as (re, im) pairs
// straight from the float4 planes, and A = sum c_k a_k is formed from two packed sums,
// (sum cr_k re_k, sum cr_k im_k) and (sum ci_k re_k, sum ci_k im_k), B likewise: four packed
// FMAs per amplitude instead of eight scalar ones.
template <int KB>
__device__ __forceinline__ void td4_sums_f32(const Td4Args<float>& a, const float2 (&am)[KB], float& Ar, float& Ai,
                                             float& Br, float& Bi) {
  using namespace pk;
  float2 P1 = splat(0.f), P2 = splat(0.f), Q1 = splat(0.f), Q2 = splat(0.f);
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    P1 = fma(splat(a.cr[k]), am[k], P1);
    P2 = fma(splat(a.ci[k]), am[k], P2);
    Q1 = fma(splat(a.br[k]), am[k], Q1);
    Q2 = fma(splat(a.bi[k]), am[k], Q2);
  }
  Ar = P1.x - P2.y;
  Ai = P1.y + P2.x;
  Br = Q1.x - Q2.y;
  Bi = Q1.y + Q2.x;
}

// Block and last-block reductions, then the FP64 combination with the normalisation terms the
// host formed from the Gram matrix (they depend on theta and the MC sample only, not on the
// events: an O(K^2) quadratic form, whose FP64 latency chain had been the last block's tail).
template <typename T, int KB, bool GRAD>
__device__ __forceinline__ void td4_finish(const Td4Args<T>& a, TdAcc<T, KB>& acc, int64_t begin, int64_t end,
                                           float2* partials, unsigned* counters, double* result, int out_mode,
                                           ddf* s_red, unsigned* s_bad) {
  constexpr int NS = TdLanes<KB, GRAD>::NS;
  ddf v[NS];
  v[0] = acc.lf;
  if constexpr (GRAD) {
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      v[1 + 2 * k] = (sizeof(T) == 4) ? ddf{(float)acc.lre[k], 0.f} : dd_from_double((double)acc.lre[k]);
      v[2 + 2 * k] = (sizeof(T) == 4) ? ddf{(float)acc.lim[k], 0.f} : dd_from_double((double)acc.lim[k]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      v[1 + 2 * KB + j] = (sizeof(T) == 4) ? ddf{(float)acc.lt[j], 0.f} : dd_from_double((double)acc.lt[j]);
  }
  unsigned bad = acc.bad;
  for (int m = 16; m > 0; m >>= 1) bad += __shfl_xor_sync(0xffffffffu, bad, m);
  if ((threadIdx.x & 31) == 0) s_bad[threadIdx.x >> 5] = bad;
  block_reduce_to_partials<NS>(v, NS, partials, s_red);
  if (threadIdx.x == 0) {
    unsigned b = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) b += s_bad[w];
    if (b) atomicAdd(counters + 1, b);
  }
  __shared__ double s_out[NS];
  if (!last_block_ticket(counters, gridDim.x)) return;
  // every other block added to these words before its ticket (and a fence): plain L2 reads,
  // issued before the reduction so that their latency overlaps it
  unsigned nbad = 0u, status = 0u;
  if (threadIdx.x == 0) {
    nbad = __ldcg(counters + 1);
    status = __ldcg(counters + kStatusWord);
  }
  reduce_partials(partials, NS, gridDim.x, s_out, s_red, blockDim.x);
  const double nev = (double)(end - begin);
  const int K = a.K;
  const int P = a.n_params;
  const int off = out_mode == 0 ? 2 : 3;
  // one thread per amplitude and time parameter forms its terms, then one per parameter gathers
  if constexpr (GRAD) {
    __shared__ double s_term[2 * kTdMaxAmp + 4];
    if ((int)threadIdx.x < K) {
      const int k = threadIdx.x;
      s_term[2 * k] = fma(nev, a.nrm_ur[k], -s_out[1 + 2 * k]);
      s_term[2 * k + 1] = fma(-nev, a.nrm_ui[k], -s_out[2 + 2 * k]);
    } else if (threadIdx.x >= 32 && threadIdx.x < 36) {
      const int j = threadIdx.x - 32;
      s_term[2 * kTdMaxAmp + j] = (j < 3 ? nev * a.nrm_dt[j] : 0.0) -
                                  time_gradient(j, (double)a.G, (double)a.x, (double)a.y, (double)a.s, s_out + 1 + 2 * KB, nev);
    }
    __syncthreads();
    for (int p = threadIdx.x; p < P; p += blockDim.x) result[off + p] = a.map.gather(p, s_term);
  } else {
    for (int p = threadIdx.x; p < P; p += blockDim.x) result[off + p] = 0.0;
  }
  if (threadIdx.x == 0) {
    counters[1] = 0u;
    counters[kStatusWord] = 0u;
    *counters = 0u;  // the ticket
    const double nb = status ? -1.0 : (double)nbad;  // a wait that gave up: negative count
    result[0] = -s_out[0] + nev * a.nrm_logN;
    if (out_mode == 0) {
      result[1] = nb;
      result[2 + P] = a.nrm_N;
    } else {
      result[1] = 0.0;
      result[2] = nb;
    }
  }
  result_complete(result);
}

// The FP64 sums A = sum c_k a_k and B = sum b_k a_k of event i; B comes from the cache where it holds it.
__device__ __forceinline__ void td4_sums(const Td4Args<double>& a, const double2* __restrict__ cache, int KB, int64_t i,
                                         double& Ar, double& Ai, double& Br, double& Bi) {
  Ar = Ai = Br = Bi = 0.0;
  if (a.has_b) {
    const double2 v = cache[(int64_t)a.K * a.n_total + i];
    Br = v.x;
    Bi = v.y;
  }
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    if (k >= a.K) break;
    const double2 v = cache[(int64_t)k * a.n_total + i];
    Ar = fma(a.cr[k], v.x, fma(-a.ci[k], v.y, Ar));
    Ai = fma(a.cr[k], v.y, fma(a.ci[k], v.x, Ai));
  }
  if (!a.has_b)
#pragma unroll 1
    for (int k = 0; k < a.K; ++k) td4_add_b(a.br[k], a.bi[k], cache[(int64_t)k * a.n_total + i], Br, Bi);
}

// FP64: direct loads, one event per thread per grid-stride step.  Bound by the FP64 pipe's slots
// (fp64.cuh): FMA chains, exp and erfcx from tables in shared memory, the logarithm as a running
// product, tests on the integer pipe.  The amplitudes are read again for the gradient lanes
// (their registers would spill; the second read costs no FP64 slot).  1M events, 10 amplitudes with
// the gradient: 872 -> 571 us (three slots per product pair and CUDA's exp, erfcx, log and division
// before), 500 us with B from the cache.
template <int KB, bool GRAD>
__global__ void __launch_bounds__(kBlock, 2) td4_nll_f64_kernel(const __grid_constant__ Td4Args<double> a,
                                                                const double2* __restrict__ cache,
                                                                const double* __restrict__ tcol,
                                                                const Fp64Tables* __restrict__ tables, int64_t begin,
                                                                int64_t end, float2* partials, unsigned* counters,
                                                                double* result, int out_mode) {
  constexpr int NS = TdLanes<KB, GRAD>::NS;
  __shared__ ddf s_red[(kBlock / 32) * NS > kBlock ? (kBlock / 32) * NS : kBlock];
  __shared__ unsigned s_bad[kBlock / 32];
  __shared__ TimeTables s_tab;
  load_fp64_tables(s_tab, tables);
  const TdMath<double> F{s_tab};
  TdAcc<double, KB> acc;
  LogProduct lp;
  double lf64 = 0.0;
#pragma unroll
  for (int k = 0; k < KB; ++k) acc.lre[k] = acc.lim[k] = 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) acc.lt[j] = 0.0;
  const int64_t n = a.n_total;
  __syncthreads();
  for (int64_t i = begin + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < end;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double t = tcol[i];
    double Ar, Ai, Br, Bi;
    td4_sums(a, cache, KB, i, Ar, Ai, Br, Bi);
    TimeTerms<double> tt;
    time_terms_g<double>(F, a.tc, a.wa, a.wN, a.wL, t, tt);
    const double AA = fma_rn(Ar, Ar, mul_rn(Ai, Ai)), BB = fma_rn(Br, Br, mul_rn(Bi, Bi));
    const double ABr = fma_rn(Ar, Br, mul_rn(Ai, Bi)), ABi = fma_rn(Ai, Br, -mul_rn(Ar, Bi));  // A conj(B)
    const double R = td_rate(tt, AA, BB, ABr, ABi);
    double invR;
    if (positive_normal(R)) {
      lp.mul(R);
      invR = rcp64(R);
    } else if (R > 0.0) {  // subnormal or infinite
      lf64 += log(R);
      invR = 1.0 / R;
    } else {
      acc.bad++;
      continue;
    }
    if constexpr (GRAD) {
      // V / R, V = (T_ch + T_c) A* + (T_sh - i T_s) B* = 2 P A* + (T_sh - i T_s) B*
      const double c1 = 2.0 * tt.P * invR, sh = tt.Tsh * invR, ss = tt.Ts * invR;
      const double Vr = fma(c1, Ar, fma(sh, Br, -ss * Bi));
      const double mVi = fma(c1, Ai, fma(sh, Bi, ss * Br));  // -Im V / R
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        if (k >= a.K) break;
        const double2 v = cache[(int64_t)k * n + i];
        acc.lre[k] = fma(v.x, Vr, fma(v.y, mVi, acc.lre[k]));   // Re(a_k V) / R
        acc.lim[k] = fma(v.x, mVi, fma(-v.y, Vr, acc.lim[k]));  // -Im(a_k V) / R
      }
      time_lanes(a.tc, t, tt, AA, BB, ABr, ABi, invR, acc.lt);
    }
  }
  acc.lf = dd_from_double(lf64 + lp.log_value());
  td4_finish<double, KB, GRAD>(a, acc, begin, end, partials, counters, result, out_mode, s_red, s_bad);
}

// FP32: tiles of kTdTile events (aligned to multiples of kTdTile) of every amplitude plane
// and of the time column staged in shared memory by bulk copies, kTdStages tiles ahead, the warps
// releasing the stages one by one (TileRing);
// block b takes tiles tb0 + b, + gridDim.x, ...; ragged first / last tiles read global
// memory.  A thread takes events e and e + kBlock of a tile: what depends on the time (exp, erfcx, the
// moment series, the rate and its derivatives, 280 of the 500 instructions an event took one at
// a time) runs once for both in packed FP32, and two events' independent sums overlap.  The
// amplitudes are read from the tile again for the gradient lanes, as packed
//   G1_k += Re(V/R) a_k,  G2_k += Im(V/R) a_k   (Re(a_k V)/R = G1.x - G2.y, Im = G1.y + G2.x).
// log2 R is summed, scaled by ln 2 once per thread; 1/R is the hardware reciprocal.
// 2M events, 10 amplitudes: 52.4 us one event at a time, now 45.6 us (84 bytes per event: 24.8 us of HBM).
// Dynamic shared memory: kTdStages * (planes * kTdTile float4 + kTdTile float).
constexpr int kTdTile = 2 * kBlock;
// stages by slot count: two blocks per SM at 10 amplitudes (43 KB a stage), one at 16 (68 KB)
template <int KB>
constexpr int kTdStages = KB <= 10 ? 2 : 3;

template <int KB, bool GRAD>
__global__ void __launch_bounds__(kBlock, KB <= 10 ? 2 : 1)
    td4_nll_f32_kernel(const __grid_constant__ Td4Args<float> a, const float4* __restrict__ cache,
                       const float* __restrict__ tcol, const Fp32Tables* __restrict__ tables, int64_t begin, int64_t end,
                       float2* partials, unsigned* counters, double* result, int out_mode) {
  using namespace pk;
  constexpr int NS = TdLanes<KB, GRAD>::NS;
  constexpr int TE = kTdTile, NST = kTdStages<KB>;
  __shared__ ddf s_red[(kBlock / 32) * NS > kBlock ? (kBlock / 32) * NS : kBlock];
  __shared__ unsigned s_bad[kBlock / 32];
  __shared__ __align__(8) TileRing<NST> s_ring;
  __shared__ Fp32Tables s_tab;
  extern __shared__ __align__(128) float4 s_tile[];  // per stage: planes x TE float4, then TE float
  const int planes = a.planes;
  const int64_t n = a.n_total;
  const size_t stage_f4 = (size_t)planes * TE + TE / 4;
  const int64_t tb0 = begin / TE, tb1 = (end + TE - 1) / TE;
  auto tile_of = [&](int j) { return tb0 + blockIdx.x + (int64_t)j * gridDim.x; };
  auto full = [&](int64_t t) { return t * TE >= begin && (t + 1) * TE <= end; };
  auto issue = [&](int j) {
    const int64_t t = tile_of(j);
    if (t >= tb1) return;
    uint64_t* bar = &s_ring.bar[j % NST];
    s_ring.last[j % NST] = j;
    float4* base = s_tile + (size_t)(j % NST) * stage_f4;
    if (full(t)) {
      mbar_arrive_expect_tx(bar, (unsigned)(planes * TE * sizeof(float4) + TE * sizeof(float)));
      for (int p = 0; p < planes; ++p) bulk_load(base + (size_t)p * TE, cache + (int64_t)p * n + t * TE, TE * sizeof(float4), bar);
      bulk_load(base + (size_t)planes * TE, tcol + t * TE, TE * sizeof(float), bar);
    } else {
      mbar_arrive(bar);
    }
  };
  if (threadIdx.x == 0) {
    s_ring.init();
    for (int j = 0; j < NST; ++j) issue(j);
  }
  for (int i = threadIdx.x; i < (int)(sizeof(Fp32Tables) / 4); i += kBlock)
    ((float*)&s_tab)[i] = __ldg((const float*)tables + i);
  const TdMath<float2> F{s_tab};
  Kahan2 lf;
  float2 G1[KB], G2[KB], lt[4];
#pragma unroll
  for (int k = 0; k < KB; ++k) G1[k] = G2[k] = splat(0.f);
#pragma unroll
  for (int j = 0; j < 4; ++j) lt[j] = splat(0.f);
  unsigned bad = 0;
  // two events: load(e, p) is plane p of event e (0, 1), t their times, v0, v1 whether they count
  auto pair = [&](auto load, float2 t, bool v0, bool v1) {
    float Ar[2], Ai[2], Br[2], Bi[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float2 P1 = splat(0.f), P2 = splat(0.f), Q1 = splat(0.f), Q2 = splat(0.f);
#pragma unroll
      for (int p = 0; p < KB / 2; ++p) {
        if (p >= planes) break;
        const float4 v = load(e, p);
        const float2 a0 = make_float2(v.x, v.y), a1 = make_float2(v.z, v.w);
        P1 = fma(splat(a.cr[2 * p + 1]), a1, fma(splat(a.cr[2 * p]), a0, P1));
        P2 = fma(splat(a.ci[2 * p + 1]), a1, fma(splat(a.ci[2 * p]), a0, P2));
        Q1 = fma(splat(a.br[2 * p + 1]), a1, fma(splat(a.br[2 * p]), a0, Q1));
        Q2 = fma(splat(a.bi[2 * p + 1]), a1, fma(splat(a.bi[2 * p]), a0, Q2));
      }
      Ar[e] = P1.x - P2.y;
      Ai[e] = P1.y + P2.x;
      Br[e] = Q1.x - Q2.y;
      Bi[e] = Q1.y + Q2.x;
    }
    const float2 A2r = make_float2(Ar[0], Ar[1]), A2i = make_float2(Ai[0], Ai[1]);
    const float2 B2r = make_float2(Br[0], Br[1]), B2i = make_float2(Bi[0], Bi[1]);
    TimeTerms<float2> tt;
    time_terms_pair(F, a.tc, a.wa, a.wN, a.wL, t, tt);
    const float2 AA = fma_rn(A2r, A2r, mul_rn(A2i, A2i)), BB = fma_rn(B2r, B2r, mul_rn(B2i, B2i));
    const float2 ABr = fma_rn(A2r, B2r, mul_rn(A2i, B2i)), ABi = sub_rn(mul_rn(A2i, B2r), mul_rn(A2r, B2i));  // A conj(B)
    const float2 R = td_rate(tt, AA, BB, ABr, ABi);
    const bool ok0 = v0 && R.x > 0.f, ok1 = v1 && R.y > 0.f;
    bad += (unsigned)(v0 && !ok0) + (unsigned)(v1 && !ok1);
    lf.add(make_float2(ok0 ? lg2(R.x) : 0.f, ok1 ? lg2(R.y) : 0.f));
    if constexpr (GRAD) {
      const float2 invR = make_float2(ok0 ? rcp(R.x) : 0.f, ok1 ? rcp(R.y) : 0.f);
      // V / R, V = (T_ch + T_c) A* + (T_sh - i T_s) B* = 2 P A* + (T_sh - i T_s) B*; mVi = -Im V / R
      const float2 c1 = mul_rn(mul_rn(splat(2.f), tt.P), invR), sh = mul_rn(tt.Tsh, invR), ss = mul_rn(tt.Ts, invR);
      const float2 Vr = sub_rn(fma_rn(c1, A2r, mul_rn(sh, B2r)), mul_rn(ss, B2i));
      const float2 mVi = fma_rn(c1, A2i, fma_rn(sh, B2i, mul_rn(ss, B2r)));
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float2 vr = splat(e ? Vr.y : Vr.x), vi = splat(e ? -mVi.y : -mVi.x);
#pragma unroll
        for (int p = 0; p < KB / 2; ++p) {
          if (p >= planes) break;
          const float4 v = load(e, p);
          const float2 a0 = make_float2(v.x, v.y), a1 = make_float2(v.z, v.w);
          G1[2 * p] = fma(vr, a0, G1[2 * p]);
          G2[2 * p] = fma(vi, a0, G2[2 * p]);
          G1[2 * p + 1] = fma(vr, a1, G1[2 * p + 1]);
          G2[2 * p + 1] = fma(vi, a1, G2[2 * p + 1]);
        }
      }
      time_lanes(a.tc, t, tt, AA, BB, ABr, ABi, invR, lt);
    }
  };
  __syncthreads();  // barriers initialised and the table copied before any thread uses them
  const long long wlim = tile_wait_limit(counters);
  bool gave_up = false;
  for (int j = 0; tile_of(j) < tb1; ++j) {
    const int64_t t = tile_of(j);
    if (!s_ring.wait(j, wlim)) {
      gave_up = true;
      break;
    }
    if (full(t)) {
      const float4* sb = s_tile + (size_t)(j % NST) * stage_f4 + threadIdx.x;
      const float* st = reinterpret_cast<const float*>(s_tile + (size_t)(j % NST) * stage_f4 + (size_t)planes * TE) + threadIdx.x;
      pair([&](int e, int p) { return sb[(size_t)p * TE + e * kBlock]; }, make_float2(st[0], st[kBlock]), true, true);
    } else {
      const int64_t i0 = t * TE + threadIdx.x, i1 = i0 + kBlock;
      const bool v0 = i0 >= begin && i0 < end, v1 = i1 >= begin && i1 < end;
      // an event outside the range takes the other's place, with weight 0
      if (v0 || v1) {
        const int64_t j0 = v0 ? i0 : i1, j1 = v1 ? i1 : i0;
        pair([&](int e, int p) { return __ldg(cache + (int64_t)p * n + (e ? j1 : j0)); },
             make_float2(__ldg(tcol + j0), __ldg(tcol + j1)), v0, v1);
      }
    }
    s_ring.release(j, issue);
  }
  s_ring.finish(gave_up, counters);
  TdAcc<float, KB> acc;
  acc.lf = dd_mul(lf.value(), ddf{kLn2Hi, kLn2Lo});
  acc.bad = bad;
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    acc.lre[k] = G1[k].x - G2[k].y;
    acc.lim[k] = -(G1[k].y + G2[k].x);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) acc.lt[j] = lt[j].x + lt[j].y;
  td4_finish<float, KB, GRAD>(a, acc, begin, end, partials, counters, result, out_mode, s_red, s_bad);
}

// per-event log f = log R - log N (goo_eval_logf)
template <int KB>
__global__ void td4_logf_f32_kernel(const __grid_constant__ Td4Args<float> a, const float4* __restrict__ cache,
                                    const float* __restrict__ tcol, double logN, double* __restrict__ out) {
  const int64_t n = a.n_total;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float2 am[KB];
#pragma unroll
    for (int p = 0; p < KB / 2; ++p) {
      const float4 v = p < a.planes ? cache[(int64_t)p * n + i] : make_float4(0.f, 0.f, 0.f, 0.f);
      am[2 * p] = make_float2(v.x, v.y);
      am[2 * p + 1] = make_float2(v.z, v.w);
    }
    float Ar, Ai, Br, Bi;
    td4_sums_f32(a, am, Ar, Ai, Br, Bi);
    TimeTerms<float> tt;
    time_terms_g<float>(TdMath<float>{}, a.tc, a.wa, a.wN, a.wL, tcol[i], tt);
    const float R = td_rate(tt, fma_rn(Ar, Ar, mul_rn(Ai, Ai)), fma_rn(Br, Br, mul_rn(Bi, Bi)),
                            fma_rn(Ar, Br, mul_rn(Ai, Bi)), fma_rn(Ai, Br, -mul_rn(Ar, Bi)));
    out[i] = R > 0.f ? (double)logf(R) - logN : -HUGE_VAL;
  }
}

template <int KB>
__global__ void td4_logf_f64_kernel(const __grid_constant__ Td4Args<double> a, const double2* __restrict__ cache,
                                    const double* __restrict__ tcol, const Fp64Tables* __restrict__ tables, double logN,
                                    double* __restrict__ out) {
  __shared__ TimeTables s_tab;
  load_fp64_tables(s_tab, tables);
  __syncthreads();
  const int64_t n = a.n_total;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double Ar, Ai, Br, Bi;
    td4_sums(a, cache, KB, i, Ar, Ai, Br, Bi);
    TimeTerms<double> tt;
    time_terms_g<double>(TdMath<double>{s_tab}, a.tc, a.wa, a.wN, a.wL, tcol[i], tt);
    const double R = td_rate(tt, fma_rn(Ar, Ar, mul_rn(Ai, Ai)), fma_rn(Br, Br, mul_rn(Bi, Bi)),
                             fma_rn(Ar, Br, mul_rn(Ai, Bi)), fma_rn(Ai, Br, -mul_rn(Ar, Bi)));
    out[i] = R > 0.0 ? log(R) - logN : -HUGE_VAL;
  }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
struct Td4Model {
  int K = 0;
  int par_re[kTdMaxAmp], par_im[kTdMaxAmp], par_t[4];
  double br[kTdMaxAmp], bi[kTdMaxAmp];
  Td4Dev host{};
  Td4Dev* dev = nullptr;
  double gram_host[2][kTdMaxAmp * kTdMaxAmp * 2];
  uint64_t gram_key[2] = {0, 0};
  const goo_dataset* mc = nullptr;
  uint64_t key = 0;
};

static double two_body_q(double m, double ma, double mb) {
  const double lam = (m * m - (ma + mb) * (ma + mb)) * (m * m - (ma - mb) * (ma - mb));
  return std::sqrt(lam > 0 ? lam : 0.0) / (2.0 * m);
}

static double barrier_host(int L, double z) {
  if (L == 0) return 1.0;
  if (L == 1) return std::sqrt(1.0 / (1.0 + z));
  return std::sqrt(9.0 / (9.0 + 3.0 * z + z * z));
}

static void spins_of(int ang, int& L1, int& L2) {
  static const int s1[8] = {0, 1, 0, 1, 1, 1, 2, 2}, s2[8] = {0, 0, 1, 1, 1, 1, 0, 1};
  L1 = s1[ang];
  L2 = s2[ang];
}

int build_td4_model(goo_ctx* ctx, const goo_node* nodes, int n_nodes, int n_params, int n_obs, goo_model* m) {
  const goo_node& root = nodes[n_nodes - 1];
  if (n_obs != 6) return set_error(GOO_ERR_ARG, "GOO_OP_TD4 needs the 6 observables m12, m34, c12, c34, phi, t");
  if (root.n_child < 1 || root.n_child > kTdMaxAmp)
    return set_error(GOO_ERR_UNSUPPORTED, "GOO_OP_TD4 with %d amplitudes (1..%d)", root.n_child, kTdMaxAmp);
  Td4Model* d = new Td4Model();
  m->td4 = d;
  m->kind = 2;
  Td4Dev& h = d->host;
  h.K = d->K = root.n_child;
  h.m1 = root.dval[1];
  h.m2 = root.dval[2];
  h.m3 = root.dval[3];
  h.m4 = root.dval[4];
  h.r = root.dval[5];
  const double M = root.dval[0];
  if (!(M > h.m1 + h.m2 + h.m3 + h.m4) || h.r < 0)
    return set_error(GOO_ERR_ARG, "GOO_OP_TD4: parent mass below threshold or negative barrier radius");
  for (int j = 0; j < 4; ++j) {
    if (root.par[j] < 0 || root.par[j] >= n_params)
      return set_error(GOO_ERR_ARG, "GOO_OP_TD4: time parameter %d has index %d", j, root.par[j]);
    d->par_t[j] = root.par[j];
  }
  for (int k = 0; k < d->K; ++k) {
    const goo_node& a = nodes[root.child[k]];
    if (a.op != GOO_OP_AMP4) return set_error(GOO_ERR_ARG, "GOO_OP_TD4 child %d is not GOO_OP_AMP4", k);
    if (a.ival[0] < GOO_ANG_SS || a.ival[0] > GOO_ANG_TV0) return set_error(GOO_ERR_ARG, "angular type %d", a.ival[0]);
    for (int j = 0; j < 2; ++j)
      if (a.par[j] < 0 || a.par[j] >= n_params) return set_error(GOO_ERR_ARG, "amplitude %d coefficient index", k);
    d->par_re[k] = a.par[0];
    d->par_im[k] = a.par[1];
    h.br[k] = d->br[k] = a.dval[4];
    h.bi[k] = d->bi[k] = a.dval[5];
    Td4Amp& A = h.amp[k];
    A.ang = a.ival[0];
    spins_of(A.ang, A.L1, A.L2);
    A.m0a = a.dval[0];
    A.g0a = a.dval[1];
    A.m0b = a.dval[2];
    A.g0b = a.dval[3];
    if (!(A.m0a > h.m1 + h.m2) || !(A.m0b > h.m3 + h.m4) || !(A.g0a > 0) || !(A.g0b > 0))
      return set_error(GOO_ERR_ARG, "amplitude %d: resonance below its pair threshold or width <= 0", k);
    A.q0a = two_body_q(A.m0a, h.m1, h.m2);
    A.q0b = two_body_q(A.m0b, h.m3, h.m4);
    A.b0a = barrier_host(A.L1, (h.r * A.q0a) * (h.r * A.q0a));
    A.b0b = barrier_host(A.L2, (h.r * A.q0b) * (h.r * A.q0b));
  }
  uint64_t key = 1469598103934665603ull;  // FNV-1a over the cache's constants
  const unsigned char* bytes = (const unsigned char*)&h;
  for (size_t i = 0; i < sizeof(Td4Dev); ++i) key = (key ^ bytes[i]) * 1099511628211ull;
  d->key = key;
  if (cudaMalloc(&d->dev, sizeof(Td4Dev)) != cudaSuccess) {
    cudaGetLastError();
    return set_error(GOO_ERR_OOM, "goo_model_build: four-body model tables");
  }
  GOO_CUDA_TRY(cudaMemcpyAsync(d->dev, &h, sizeof(Td4Dev), cudaMemcpyHostToDevice, ctx->stream));
  GOO_CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  (void)weideman();
  return GOO_OK;
}

void td4_free(goo_model* m) {
  Td4Model* d = m->td4;
  if (!d) return;
  if (d->dev) cudaFree(d->dev);
  delete d;
  m->td4 = nullptr;
}

int td4_set_norm(goo_model* m, const goo_norm_spec* spec) {
  if (spec->kind != GOO_NORM_MC || !spec->mc)
    return set_error(GOO_ERR_UNSUPPORTED, "the four-body model is normalised with GOO_NORM_MC and a phase-space sample");
  if (spec->mc->ncols < 5) return set_error(GOO_ERR_ARG, "the MC sample needs the five phase-space columns");
  m->td4->mc = spec->mc;
  m->td4->gram_key[0] = m->td4->gram_key[1] = 0;
  m->norm = *spec;
  return GOO_OK;
}

// Bytes of the FP64 cache with B's plane.
static size_t td4_bytes_b(const Td4Model& d, int64_t n) { return (size_t)(d.K + 1) * (size_t)n * sizeof(double2); }

// with_b: keep B in the FP64 cache where there is room (the events; nothing reads it from the MC sample's)
static int td4_cache(goo_model* m, const goo_dataset* ds_c, int precision, bool with_b, const void** out) {
  goo_dataset* ds = const_cast<goo_dataset*>(ds_c);
  Td4Model& d = *m->td4;
  goo_ctx* ctx = m->ctx;
  const int pi = precision == GOO_F32 ? 0 : 1;
  const uint64_t key = d.key ^ (uint64_t)(uintptr_t)m ^ (uint64_t)(pi + 3) * 0x9e3779b97f4a7c15ull ^
                       ds->epoch * 0xd6e8feb86659fd93ull;
  CacheSlot& slot = ds->cache[pi];
  const int64_t n = ds->n;
  const size_t bytes = pi == 0 ? (size_t)((d.K + 1) / 2) * (size_t)n * sizeof(float4) : (size_t)d.K * (size_t)n * sizeof(double2);
  const bool same = slot.ptr && slot.key == key && slot.bytes >= bytes;
  if (same && (pi == 0 || !with_b || slot.asked_b)) {
    *out = slot.ptr;
    return GOO_OK;
  }
  // same: an MC sample's cache that is now evaluated as events
  if (!slot.ptr || slot.bytes < bytes || same) {
    if (slot.ptr) cudaFree(slot.ptr);
    slot.ptr = nullptr;
    slot.bytes = 0;
    size_t got = pi == 1 && with_b ? td4_bytes_b(d, n) : bytes;
    cudaError_t e = cudaMalloc(&slot.ptr, got > 0 ? got : 16);
    if (e != cudaSuccess && got > bytes) {  // no room for B's plane: the evaluation forms B itself
      cudaGetLastError();
      got = bytes;
      e = cudaMalloc(&slot.ptr, got);
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      slot.ptr = nullptr;
      return set_error(GOO_ERR_OOM, "amplitude cache of %zu bytes does not fit", bytes);
    }
    slot.bytes = got;
  }
  slot.asked_b = with_b;
  slot.has_b = pi == 1 && with_b && slot.bytes >= td4_bytes_b(d, n);
  if (n > 0) {
    const int nb = grid_blocks(ctx, n, 4);
    if (pi == 0) {
      Td4Cols<float> c{};
      for (int j = 0; j < 5; ++j) c.c[j] = ds->d32[j];
      LaunchScope ls(ctx, "td4_cache_f32");
      td4_cache_kernel<float><<<nb, kBlock, 0, ctx->stream>>>(d.dev, c, n, slot.ptr, false);
    } else {
      Td4Cols<double> c{};
      for (int j = 0; j < 5; ++j) c.c[j] = ds->d64[j];
      LaunchScope ls(ctx, "td4_cache_f64");
      td4_cache_kernel<double><<<nb, kBlock, 0, ctx->stream>>>(d.dev, c, n, slot.ptr, slot.has_b);
    }
    GOO_CUDA_TRY(cudaGetLastError());
  }
  slot.key = key;
  *out = slot.ptr;
  return GOO_OK;
}

static int td4_ensure_gram(goo_model* m, int precision) {
  Td4Model& d = *m->td4;
  const int pi = precision == GOO_F32 ? 0 : 1;
  if (!d.mc) return set_error(GOO_ERR_STATE, "the four-body model has no MC normalisation sample (goo_model_set_norm)");
  if (d.K > 15) return set_error(GOO_ERR_UNSUPPORTED, "the Gram matrix supports at most 15 amplitudes");
  const uint64_t key = d.key ^ (uint64_t)(uintptr_t)d.mc ^ (uint64_t)(pi + 11) ^ d.mc->epoch * 0xd6e8feb86659fd93ull;
  if (d.gram_key[pi] == key) return GOO_OK;
  if (d.mc->n < 1) return set_error(GOO_ERR_ARG, "the MC normalisation sample is empty");
  const void* cache = nullptr;
  GOO_TRY(td4_cache(m, d.mc, precision, false, &cache));
  GOO_TRY(gram_matrices(m->ctx, precision, false, 1, &cache, &cache, d.mc->n, d.K, d.K, d.gram_host[pi],
                        pi == 0 ? "td4_gram_f32" : "td4_gram_f64"));
  d.gram_key[pi] = key;
  return GOO_OK;
}

template <typename T>
static void td4_args(const goo_model* m, const double* theta, int64_t n_total, Td4Args<T>& a) {
  const Td4Model& d = *m->td4;
  std::memset(&a, 0, sizeof a);
  a.K = d.K;
  a.planes = (d.K + 1) / 2;
  a.n_params = m->n_params;
  a.n_total = n_total;
  for (int k = 0; k < d.K; ++k) {
    a.cr[k] = (T)theta[d.par_re[k]];
    a.ci[k] = (T)theta[d.par_im[k]];
    a.br[k] = (T)d.br[k];
    a.bi[k] = (T)d.bi[k];
  }
  a.map.clear();
  for (int j = 3; j >= 0; --j) a.map.add(2 * kTdMaxAmp + j, d.par_t[j]);
  for (int k = d.K - 1; k >= 0; --k) {
    a.map.add(2 * k + 1, d.par_im[k]);
    a.map.add(2 * k, d.par_re[k]);
  }
  fill_time_coef<T>(a.tc, theta[d.par_t[0]], theta[d.par_t[1]], theta[d.par_t[2]], theta[d.par_t[3]], m->hi[5]);
  a.x = a.tc.x;
  a.y = a.tc.y;
  a.G = a.tc.G;
  a.s = a.tc.s;
  const WeidemanTables& w = weideman();
  a.wN = sizeof(T) == 4 ? kWN32 : kWN64;
  for (int j = 0; j < a.wN; ++j) a.wa[j] = (T)(sizeof(T) == 4 ? w.a32[j] : w.a64[j]);
  a.wL = (T)(sizeof(T) == 4 ? w.L32 : w.L64);
}

// The normalisation at theta from the host copy of the Gram matrix (td4_ensure_gram keeps it
// current), in FP64 and at the precision-rounded parameters the kernel uses:
//   v_c = G conj(c), v_b = G conj(b),  <|A|^2> = Re c.v_c, <|B|^2> = Re b.v_b, <A B*> = c.v_b,
//   N = <|A|^2+|B|^2>/2 I_ch + <|A|^2-|B|^2>/2 I_c + Re<AB*> I_sh + Im<AB*> I_s,
//   dN / d Re c_k = Re((I_ch + I_c) v_c,k + (I_sh - i I_s) v_b,k), dN / d Im c_k = -Im(same),
// with the time integrals' derivatives for x, y and tau.
template <typename T>
static void td4_norm_terms(const goo_model* m, int precision, Td4Args<T>& a) {
  const Td4Model& d = *m->td4;
  const int pi = precision == GOO_F32 ? 0 : 1;
  const int K = d.K;
  const double x = (double)a.x, y = (double)a.y, tau = 1.0 / (double)a.G;
  const double iy = 1.0 / (1 - y * y), ix = 1.0 / (1 + x * x);
  const double Ich = tau * iy, Ish = y * tau * iy, Ic = tau * ix, Is = x * tau * ix;
  double vcr[kTdMaxAmp], vci[kTdMaxAmp], vbr[kTdMaxAmp], vbi[kTdMaxAmp];
  double aa = 0, bb = 0, abr = 0, abi = 0;
  for (int k = 0; k < K; ++k) {
    vcr[k] = vci[k] = vbr[k] = vbi[k] = 0.0;
    for (int l = 0; l < K; ++l) {
      const double gr = d.gram_host[pi][2 * (k * K + l)], gi = d.gram_host[pi][2 * (k * K + l) + 1];
      const double clr = (double)a.cr[l], cli = (double)a.ci[l], blr = (double)a.br[l], bli = (double)a.bi[l];
      vcr[k] += gr * clr + gi * cli;  // G_kl conj(c_l)
      vci[k] += gi * clr - gr * cli;
      vbr[k] += gr * blr + gi * bli;
      vbi[k] += gi * blr - gr * bli;
    }
    const double ckr = (double)a.cr[k], cki = (double)a.ci[k], bkr = (double)a.br[k], bki = (double)a.bi[k];
    aa += ckr * vcr[k] - cki * vci[k];  // Re(c_k v_c,k)
    bb += bkr * vbr[k] - bki * vbi[k];
    abr += ckr * vbr[k] - cki * vbi[k];  // c_k v_b,k (summed: <A B*>)
    abi += ckr * vbi[k] + cki * vbr[k];
  }
  const double N = 0.5 * (aa + bb) * Ich + 0.5 * (aa - bb) * Ic + abr * Ish + abi * Is;
  const double invN = 1.0 / N;
  for (int k = 0; k < K; ++k) {
    a.nrm_ur[k] = ((Ich + Ic) * vcr[k] + Ish * vbr[k] + Is * vbi[k]) * invN;
    a.nrm_ui[k] = ((Ich + Ic) * vci[k] + Ish * vbi[k] - Is * vbr[k]) * invN;
  }
  a.nrm_N = N;
  a.nrm_logN = std::log(N);
  const double ix2 = ix * ix, iy2 = iy * iy;
  const double dxc = -2 * x * tau * ix2, dxs = tau * (1 - x * x) * ix2;
  const double dych = 2 * y * tau * iy2, dysh = tau * (1 + y * y) * iy2;
  a.nrm_dt[0] = (0.5 * (aa - bb) * dxc + abi * dxs) * invN;  // (dN/dx) / N
  a.nrm_dt[1] = (0.5 * (aa + bb) * dych + abr * dysh) * invN;
  a.nrm_dt[2] = (0.5 * (aa + bb) * iy + 0.5 * (aa - bb) * ix + abr * y * iy + abi * x * ix) * invN;  // tau dN/dtau / N
}

static int td4_check_theta(const goo_model* m, const double* theta) {
  const Td4Model& d = *m->td4;
  const double x = theta[d.par_t[0]], y = theta[d.par_t[1]], tau = theta[d.par_t[2]], s = theta[d.par_t[3]];
  if (!(tau > 0) || !(s > 0) || !(std::fabs(y) < 1) || !std::isfinite(x))
    return set_error(GOO_ERR_ARG, "four-body model: needs tau > 0, sigma_t > 0, |y| < 1 (tau=%g sigma=%g y=%g)", tau, s, y);
  return GOO_OK;
}

constexpr int kMaxDevicesTd = 64;

template <int KB, bool GRAD>
static int launch_td4_f32(goo_model* m, const void* cache, const goo_dataset* ds, int64_t begin, int64_t end,
                          const double* theta, int out_mode) {
  goo_ctx* ctx = m->ctx;
  Td4Args<float> a;
  td4_args<float>(m, theta, ds->n, a);
  td4_norm_terms<float>(m, GOO_F32, a);
  const Fp32Tables* tables = nullptr;
  GOO_TRY(fp32_tables(ctx, &tables));
  const size_t smem = (size_t)kTdStages<KB> * ((size_t)a.planes * kTdTile * sizeof(float4) + kTdTile * sizeof(float));
  static bool configured[kMaxDevicesTd] = {};
  if (ctx->device < 0 || ctx->device >= kMaxDevicesTd) return set_error(GOO_ERR_ARG, "device %d", ctx->device);
  if (!configured[ctx->device]) {
    GOO_CUDA_TRY(cudaFuncSetAttribute(td4_nll_f32_kernel<KB, GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)((size_t)kTdStages<KB> * ((KB / 2) * kTdTile * sizeof(float4) + kTdTile * sizeof(float)))));
    configured[ctx->device] = true;
  }
  const int occ = cached_occupancy((const void*)td4_nll_f32_kernel<KB, GRAD>, ctx->device, kBlock, smem);
  const int64_t tiles = (end + kTdTile - 1) / kTdTile - begin / kTdTile;
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)ctx->num_sms * occ));
  GOO_TRY(ensure_partials(ctx, (size_t)nb * TdLanes<KB, GRAD>::NS));
  {
    LaunchScope ls(ctx, GRAD ? "td4_nll_grad_f32" : "td4_nll_f32");
    td4_nll_f32_kernel<KB, GRAD><<<nb, kBlock, smem, ctx->stream>>>(a, (const float4*)cache, ds->d32[5], tables, begin, end,
                                                                   ctx->scratch.partials, ctx->scratch.counters,
                                                                   ctx->scratch.result_out, out_mode);
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

template <int KB, bool GRAD>
static int launch_td4_f64(goo_model* m, const void* cache, const goo_dataset* ds, int64_t begin, int64_t end,
                          const double* theta, int out_mode) {
  goo_ctx* ctx = m->ctx;
  Td4Args<double> a;
  td4_args<double>(m, theta, ds->n, a);
  a.has_b = ds->cache[1].has_b;
  td4_norm_terms<double>(m, GOO_F64, a);
  const Fp64Tables* tables = nullptr;
  GOO_TRY(fp64_tables(ctx, &tables));
  const int occ = cached_occupancy((const void*)td4_nll_f64_kernel<KB, GRAD>, ctx->device, kBlock, 0);
  const int nb = grid_blocks(ctx, end - begin, occ);
  GOO_TRY(ensure_partials(ctx, (size_t)nb * TdLanes<KB, GRAD>::NS));
  {
    LaunchScope ls(ctx, GRAD ? "td4_nll_grad_f64" : "td4_nll_f64");
    td4_nll_f64_kernel<KB, GRAD><<<nb, kBlock, 0, ctx->stream>>>(a, (const double2*)cache, ds->d64[5], tables, begin, end,
                                                                ctx->scratch.partials, ctx->scratch.counters,
                                                                ctx->scratch.result_out, out_mode);
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

template <bool GRAD>
static int td4_launch(goo_model* m, const void* cache, const goo_dataset* ds, int64_t begin, int64_t end,
                      const double* theta, int precision, int out_mode) {
  const bool small = m->td4->K <= 10;
  if (precision == GOO_F32)
    return small ? launch_td4_f32<10, GRAD>(m, cache, ds, begin, end, theta, out_mode)
                 : launch_td4_f32<16, GRAD>(m, cache, ds, begin, end, theta, out_mode);
  return small ? launch_td4_f64<10, GRAD>(m, cache, ds, begin, end, theta, out_mode)
               : launch_td4_f64<16, GRAD>(m, cache, ds, begin, end, theta, out_mode);
}

int td4_nll(goo_model* m, const goo_dataset* ds, int64_t begin, int64_t end, const double* theta, int precision,
            bool grad, double* out, int out_mode) {
  goo_ctx* ctx = m->ctx;
  // the record goes to the mapped host copy; the host polls its fields
  MappedResult mapped(ctx);
  const int P = m->n_params;
  if (ds->ncols < 6) return set_error(GOO_ERR_ARG, "the four-body model needs 6 dataset columns");
  GOO_TRY(td4_check_theta(m, theta));
  GOO_TRY(td4_ensure_gram(m, precision));
  const int nout = (out_mode == 0 ? 2 : 3) + P;
  if (end <= begin) {
    for (int i = 0; i < nout; ++i) out[i] = 0.0;
    return GOO_OK;
  }
  const void* cache = nullptr;
  GOO_TRY(td4_cache(m, ds, precision, true, &cache));
  GOO_TRY((grad ? td4_launch<true>(m, cache, ds, begin, end, theta, precision, out_mode)
                : td4_launch<false>(m, cache, ds, begin, end, theta, precision, out_mode)));
  return read_result_mapped(ctx, nout, out);
}

// N at theta from the host copy of the Gram matrix (the same formula as the kernels' last block)
static double td4_norm_host(const goo_model* m, const double* theta, int precision) {
  const Td4Model& d = *m->td4;
  const int pi = precision == GOO_F32 ? 0 : 1;
  const bool f32 = precision == GOO_F32;
  auto rnd = [&](double v) { return f32 ? (double)(float)v : v; };
  double aa = 0, bb = 0, abr = 0, abi = 0;
  const int K = d.K;
  for (int k = 0; k < K; ++k) {
    const double ckr = rnd(theta[d.par_re[k]]), cki = rnd(theta[d.par_im[k]]), bkr = rnd(d.br[k]), bki = rnd(d.bi[k]);
    double vcr = 0, vci = 0, vbr = 0, vbi = 0;
    for (int l = 0; l < K; ++l) {
      const double gr = d.gram_host[pi][2 * (k * K + l)], gi = d.gram_host[pi][2 * (k * K + l) + 1];
      const double clr = rnd(theta[d.par_re[l]]), cli = rnd(theta[d.par_im[l]]), blr = rnd(d.br[l]), bli = rnd(d.bi[l]);
      vcr += gr * clr + gi * cli;
      vci += gi * clr - gr * cli;
      vbr += gr * blr + gi * bli;
      vbi += gi * blr - gr * bli;
    }
    aa += ckr * vcr - cki * vci;
    bb += bkr * vbr - bki * vbi;
    abr += ckr * vbr - cki * vbi;
    abi += ckr * vbi + cki * vbr;
  }
  const double x = rnd(theta[d.par_t[0]]), y = rnd(theta[d.par_t[1]]);
  const double tau = 1.0 / rnd(1.0 / theta[d.par_t[2]]);
  return 0.5 * (aa + bb) * tau / (1 - y * y) + 0.5 * (aa - bb) * tau / (1 + x * x) + abr * y * tau / (1 - y * y) +
         abi * x * tau / (1 + x * x);
}

int td4_normalise(goo_model* m, const double* theta, int precision, double* norm_out) {
  GOO_TRY(td4_check_theta(m, theta));
  GOO_TRY(td4_ensure_gram(m, precision));
  *norm_out = td4_norm_host(m, theta, precision);
  return GOO_OK;
}

int td4_eval_logf(goo_model* m, const goo_dataset* ds, const double* theta, int precision, double* logf_dev) {
  goo_ctx* ctx = m->ctx;
  if (ds->ncols < 6) return set_error(GOO_ERR_ARG, "the four-body model needs 6 dataset columns");
  GOO_TRY(td4_check_theta(m, theta));
  GOO_TRY(td4_ensure_gram(m, precision));
  if (ds->n == 0) return GOO_OK;
  const double logN = std::log(td4_norm_host(m, theta, precision));
  const void* cache = nullptr;
  GOO_TRY(td4_cache(m, ds, precision, true, &cache));
  const int nb = grid_blocks(ctx, ds->n, 4);
  LaunchScope ls(ctx, "td4_logf");
  const bool small = m->td4->K <= 10;
  if (precision == GOO_F32) {
    Td4Args<float> a;
    td4_args<float>(m, theta, ds->n, a);
    const float4* amps = (const float4*)cache;
    if (small) td4_logf_f32_kernel<10><<<nb, kBlock, 0, ctx->stream>>>(a, amps, ds->d32[5], logN, logf_dev);
    else td4_logf_f32_kernel<16><<<nb, kBlock, 0, ctx->stream>>>(a, amps, ds->d32[5], logN, logf_dev);
  } else {
    Td4Args<double> a;
    td4_args<double>(m, theta, ds->n, a);
    a.has_b = ds->cache[1].has_b;
    const Fp64Tables* tables = nullptr;
    GOO_TRY(fp64_tables(ctx, &tables));
    const double2* amps = (const double2*)cache;
    if (small) td4_logf_f64_kernel<10><<<nb, kBlock, 0, ctx->stream>>>(a, amps, ds->d64[5], tables, logN, logf_dev);
    else td4_logf_f64_kernel<16><<<nb, kBlock, 0, ctx->stream>>>(a, amps, ds->d64[5], tables, logN, logf_dev);
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

int td4_gram(goo_model* m, int precision, double* out, int* K_out) {
  GOO_TRY(td4_ensure_gram(m, precision));
  const int pi = precision == GOO_F32 ? 0 : 1;
  std::memcpy(out, m->td4->gram_host[pi], sizeof(double) * 2 * m->td4->K * m->td4->K);
  *K_out = m->td4->K;
  return GOO_OK;
}

int td4_amplitudes(goo_model* m, const goo_dataset* ds, int precision, const void** cache, int* n_amp) {
  if (ds->ncols < 5) return set_error(GOO_ERR_ARG, "the four-body model needs the five phase-space columns");
  GOO_TRY(td4_cache(m, ds, precision, true, cache));
  GOO_CUDA_TRY(cudaStreamSynchronize(m->ctx->stream));
  *n_amp = m->td4->K;
  return GOO_OK;
}

}  // namespace goo

// Host evaluation of the library's Faddeeva approximation (the same code the kernels run),
// exposed so that it can be checked against an independent implementation on the CPU.
extern "C" int goo_faddeeva(double re, double im, int precision, double* out) {
  using namespace goo;
  if (!out) return set_error(GOO_ERR_ARG, "goo_faddeeva: NULL output");
  if (!(im >= 0.0)) return set_error(GOO_ERR_ARG, "goo_faddeeva: Im z must be >= 0");
  const WeidemanTables& w = weideman();
  if (precision == GOO_F32) {
    float a[kWMax];
    for (int j = 0; j < kWN32; ++j) a[j] = (float)w.a32[j];
    float wr, wi;
    faddeeva<float>((float)re, (float)im, a, kWN32, (float)w.L32, wr, wi);
    out[0] = wr;
    out[1] = wi;
  } else if (precision == GOO_F64) {
    double wr, wi;
    faddeeva<double>(re, im, w.a64, kWN64, w.L64, wr, wi);
    out[0] = wr;
    out[1] = wi;
  } else {
    return set_error(GOO_ERR_ARG, "goo_faddeeva: precision=%d", precision);
  }
  return GOO_OK;
}
