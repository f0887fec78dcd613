// dalitz.cu -- three-body amplitude (Dalitz-plot) models: amplitude cache, MC Gram matrix
// and the coherent-sum NLL with its adjoint gradient.
//
// Paper: GooFit carries dedicated amplitude PDFs for three-body decays (Sec. 1), whose
// components are complex amplitudes with the density given by the squared magnitude of
// their sum (Sec. 1, footnote); PDFs cache partial results in structure-of-arrays form
// and recompute them only when their parameters change (Sec. 4); MC phase-space samples
// provide the normalisation integral (Sec. 5).
//
// Model (isobar convention; the paper prints no formulas):
//   S(x) = sum_k c_k A_k(x),  f = |S|^2 / N,  N = c^H G c,  G_kl = mean over the MC sample
//   of A_k conj(A_l);  NLL = -sum_i log |S_i|^2 + n log N.
//   A_R(s12, s13) = BW(s_AB) * B_L(r q)/B_L(r q0) * B_L(r_par p*) * Z_L for resonance R in
//   pair (A, B) with bachelor C, where
//     q^2  = lambda(s, mA^2, mB^2) / (4 s),   p*^2 = lambda(M^2, s, mC^2) / (4 M^2),
//     B_0 = 1, B_1(z) = sqrt(1/(1+z)), B_2(z) = sqrt(9/(9+3z+z^2)),   z = r^2 q^2,
//     Gamma(s) = G0 (q/q0)^(2L+1) (m0/sqrt s) (B_L(z)/B_L(z0))^2,
//     BW(s) = 1 / (m0^2 - s - i m0 Gamma(s)),
//     Z_0 = 1,  Z_1 = s_AC - s_BC - (mA^2 - mB^2)(M^2 - mC^2)/s,
//     Z_2 = Z_1^2 - lambda(s, mA^2, mB^2) lambda(M^2, s, mC^2) / (3 s^2)
//   (Z_1 = -4 q k cos(theta) and Z_2 = 16 q^2 k^2 (cos^2 - 1/3) in the resonance frame).
//   lambda(s, a^2, b^2) is evaluated in its factorised form (s-(a+b)^2)(s-(a-b)^2).
//
// Gradient: d|S|^2/d Re c_k = 2 Re(A_k conj S), d|S|^2/d Im c_k = -2 Im(A_k conj S), and
// for the normalisation dN/d Re c_k = 2 Re(v_k), dN/d Im c_k = -2 Im(v_k), v = G conj(c).
// The event kernel accumulates sum_i A_k conj(S_i) / |S_i|^2 (2K lanes) and sum log|S|^2.
//
// FP32 path: amplitudes and S in FP32, Kahan per thread, double-float across threads; the
// final FP64 combination takes c at the FP32-rounded values the kernel used, so the NLL is
// the exact likelihood at those coefficients.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "dalitz.cuh"
#include "fp64.cuh"
#include "gram.cuh"
#include "lineshape.cuh"
#include "timeterms.cuh"
#include "model.cuh"

namespace goo {

struct DalitzModel {
  int K = 0;                       // amplitudes, BWs first then the NR (if any)
  int nbw = 0;
  bool has_nr = false;
  int par_re[kMaxAmp], par_im[kMaxAmp];
  int par_m0[kMaxAmp], par_w[kMaxAmp];
  int spin[kMaxAmp], pair[kMaxAmp];
  int col12 = 0, col13 = 1;
  double M = 0, m1 = 0, m2 = 0, m3 = 0, r_res = 0, r_par = 0;
  DalitzDev host{};
  DalitzDev* dev = nullptr;
  uint64_t ls_key = 0;             // lineshape version of `host` and the tables below
  uint64_t dev_key = 0;            // lineshape version of `dev` (dalitz_dev)
  LsTables<double> ls64{};         // the lineshape constants of lineshape.cuh, passed by value
  LsTables<float> ls32{};
  // Gram matrices (K x K complex, row-major, FP64) per precision, with their keys
  double gram_host[2][kMaxAmp * kMaxAmp * 2];
  uint64_t gram_key[2] = {0, 0};
  const goo_dataset* mc = nullptr;
  bool floating = false;           // GOO_LINESHAPE_FLOATING: no cache, lineshape gradients
  bool polar = false;              // GOO_COEF_POLAR: the coefficient parameters are (r, phi)
  // time-dependent three-body model (GOO_OP_TD3)
  bool td = false;
  int col_t = 2;
  int par_t[4] = {-1, -1, -1, -1};  // x, y, tau, sigma_t
  double gram3_host[2][3 * kMaxAmp * kMaxAmp * 2];  // per precision: G_aa, G_bb, G_ab (K x K complex each)
  uint64_t gram3_key[2] = {0, 0};
};

// Cache layout.  FP32: ceil(nbw/2) planes of float4 (re_k, im_k, re_k+1, im_k+1) per event;
// FP64: nbw planes of double2 (re, im) per event.  Plane p of an n-event dataset starts at
// element p * n.  FP32: two events per thread (packed arithmetic, lineshape.cuh), whose float4 of a
// plane are adjacent, so a thread writes 32 contiguous bytes per plane.  2M events of 8
// resonances: 97 us with every resonance evaluated by itself, now 34 us (144 MB moved).
// Built behind a Gram kernel, of which it needs nothing, it starts on the SMs that kernel's
// blocks leave (grid_dep_wait at the end only keeps the stream's order for what follows).
__global__ void __launch_bounds__(kLsBlock)
    amp_cache_f32_kernel(const __grid_constant__ LsTables<float> t, const float* __restrict__ s12c,
                         const float* __restrict__ s13c, int64_t n, float4* __restrict__ cache) {
  grid_dep_launch();
  __shared__ float2 s_v[kLsCols][kLsBlock];
  float2 *sc = &s_v[0][threadIdx.x], *gc = &s_v[3][threadIdx.x], *hc = &s_v[12][threadIdx.x];
  const int planes = (t.nbw + 1) / 2;
  const int64_t npair = (n + 1) / 2;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < npair; j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = 2 * j;
    const bool two = i + 1 < n;
    float2 a, b;
    if (two) {
      a = *reinterpret_cast<const float2*>(s12c + i);
      b = *reinterpret_cast<const float2*>(s13c + i);
    } else {
      a = pk::splat(s12c[i]);
      b = pk::splat(s13c[i]);
    }
    ls_groups<float, float2>(t, a, b, sc, gc, hc, kLsBlock);
    for (int p = 0; p < planes; ++p) {
      float2 r0, i0, r1 = pk::splat(0.f), i1 = pk::splat(0.f);
      ls_amp<float, float2>(t, 2 * p, sc, gc, hc, kLsBlock, r0, i0);
      if (2 * p + 1 < t.nbw) ls_amp<float, float2>(t, 2 * p + 1, sc, gc, hc, kLsBlock, r1, i1);
      float4* out = cache + (int64_t)p * n + i;
      out[0] = make_float4(r0.x, i0.x, r1.x, i1.x);
      if (two) out[1] = make_float4(r0.y, i0.y, r1.y, i1.y);
    }
  }
  grid_dep_wait();
}

__global__ void __launch_bounds__(kLsBlock)
    amp_cache_f64_kernel(const __grid_constant__ LsTables<double> t, const double* __restrict__ s12c,
                         const double* __restrict__ s13c, int64_t n, double2* __restrict__ cache) {
  grid_dep_launch();
  __shared__ double s_v[kLsCols][kLsBlock];
  double *sc = &s_v[0][threadIdx.x], *gc = &s_v[3][threadIdx.x], *hc = &s_v[12][threadIdx.x];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    ls_groups<double, double>(t, s12c[i], s13c[i], sc, gc, hc, kLsBlock);
    for (int k = 0; k < t.nbw; ++k) {
      double re, im;
      ls_amp<double, double>(t, k, sc, gc, hc, kLsBlock, re, im);
      cache[(int64_t)k * n + i] = make_double2(re, im);
    }
  }
  grid_dep_wait();
}

// ---------------------------------------------------------------------------------------
// coherent NLL (+ gradient lanes) over events [begin, end) of one dataset
// ---------------------------------------------------------------------------------------
template <typename T>
struct CohArgs {
  T cr[kMaxAmp], ci[kMaxAmp];  // coefficients (BWs first, then NR)
  int nbw, K, has_nr;
  GradMap<4 * kMaxAmp> map;    // terms 2k, 2k + 1: amplitude k's two coefficient parameters; floating
                               // lineshapes: 2K + 2k, + 1: resonance k's mass and width
  int n_params;
  int64_t n_total;             // events of the dataset (cache plane length)
  int polar;                   // the coefficient parameters are (r, phi): c = r e^{i phi}
  double jc[kMaxAmp], js[kMaxAmp], jr[kMaxAmp];  // cos phi, sin phi, r per amplitude (polar)
  // the normalisation at theta, formed on the host in FP64 from the cached Gram matrix
  // (coh_norm_terms): N, log N and 2 v_k / N with v_k = sum_l G_kl conj(c_l)
  double nrm_N, nrm_logN, nrm_vr[kMaxAmp], nrm_vi[kMaxAmp];
};

// A gradient over (Re c, Im c) of amplitude k mapped to its parameters (FP64): unchanged, or
// for polar coefficients d/dr = cos(phi) d/dRe + sin(phi) d/dIm and
// d/dphi = r (-sin(phi) d/dRe + cos(phi) d/dIm).
__device__ __forceinline__ void coef_chain(int polar, double c, double s, double r, double& gre, double& gim) {
  if (!polar) return;
  const double u = c * gre + s * gim, v = r * (c * gim - s * gre);
  gre = u;
  gim = v;
}

template <typename T, int KB, bool GRAD>
struct CohLanes {
  static constexpr int NS = GRAD ? 1 + 2 * (KB + 1) : 1;
};

// Per-thread accumulators of the coherent kernels.
template <typename T, int KB>
struct CohAcc {
  Kahan lf32;
  double lf64 = 0.0;
  T gre[KB + 1], gim[KB + 1];
  unsigned bad = 0;
};

// Block and last-block reductions of the lanes, then the FP64 combination with the
// normalisation terms the host formed from the Gram matrix at the coefficients the kernel used
// (they depend on theta and the MC sample only: an O(K^2) quadratic form that would otherwise
// be an FP64 latency chain on the last block).
template <typename T, int KB, bool GRAD>
__device__ __forceinline__ void coh_finish(const CohArgs<T>& a, CohAcc<T, KB>& acc, int64_t begin, int64_t end,
                                           float2* partials, unsigned* counters, double* result, int out_mode,
                                           ddf* s_red, unsigned* s_bad) {
  constexpr int NS = CohLanes<T, KB, GRAD>::NS;
  constexpr int KA = KB + 1;
  ddf v[NS];
  v[0] = (sizeof(T) == 4) ? acc.lf32.value() : dd_from_double(acc.lf64);
  if constexpr (GRAD) {
#pragma unroll
    for (int k = 0; k < KA; ++k) {
      v[1 + 2 * k] = (sizeof(T) == 4) ? ddf{(float)acc.gre[k], 0.f} : dd_from_double((double)acc.gre[k]);
      v[2 + 2 * k] = (sizeof(T) == 4) ? ddf{(float)acc.gim[k], 0.f} : dd_from_double((double)acc.gim[k]);
    }
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
  // one thread per amplitude forms its two terms, then one per parameter gathers (GradMap)
  if constexpr (GRAD) {
    __shared__ double s_term[2 * kMaxAmp];
    if ((int)threadIdx.x < K) {
      const int k = threadIdx.x;
      const int slot = (k < a.nbw) ? k : KB;  // NR lives in the last slot
      double gre = fma(nev, a.nrm_vr[k], -2.0 * s_out[1 + 2 * slot]);
      double gim = fma(-nev, a.nrm_vi[k], 2.0 * s_out[2 + 2 * slot]);
      coef_chain(a.polar, a.jc[k], a.js[k], a.jr[k], gre, gim);
      s_term[2 * k] = gre;
      s_term[2 * k + 1] = gim;
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
    const double nll = -s_out[0] + nev * a.nrm_logN;
    // a device wait that gave up is reported as a negative event count
    const double nb = status ? -1.0 : (double)nbad;
    result[0] = nll;
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

template <typename T, int KB>
__device__ __forceinline__ void coh_coeffs(const CohArgs<T>& a, T (&cr)[KB + 1], T (&ci)[KB + 1]) {
  const int nbw = a.nbw;
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    cr[k] = k < nbw ? a.cr[k] : T(0);
    ci[k] = k < nbw ? a.ci[k] : T(0);
  }
  cr[KB] = a.has_nr ? a.cr[nbw] : T(0);
  ci[KB] = a.has_nr ? a.ci[nbw] : T(0);
}

// FP64 form: one event per thread per grid-stride step, amplitudes read directly.  Bound by the
// FP64 pipe (fp64.cuh), so what counts is its slots per event: 8 per resonance (every product
// sum is a chain of FMAs), the logarithm as a running product, the reciprocal by one third-order
// step, the sign test on the integer pipe; absent resonance slots and the constant amplitude
// (A = 1) cost no multiplication.  8 resonances with the gradient take 78 slots per event; 2M
// events: 549 -> 286 us (the slots alone: 249 us at the measured 6.27e11 FMA/s).  One block per SM: with the
// registers of 16 warps to interleave independent chains 8 warps fill the pipe (286 us; 290 us with two
// blocks, 303 with 20 warps), and a small dataset's events spread over the SMs more evenly (100k: 41 -> 33 us).
template <int KB, bool GRAD>
__global__ void __launch_bounds__(kBlock, 1)
    coh_nll_f64_kernel(const __grid_constant__ CohArgs<double> a, const double2* __restrict__ cache, int64_t begin,
                       int64_t end, float2* partials, unsigned* counters, double* result, int out_mode) {
  constexpr int NS = CohLanes<double, KB, GRAD>::NS;
  constexpr int KA = KB + 1;  // BW slots + NR slot
  // the amplitudes of an event stay in registers between the sum and the gradient lanes; the
  // 15-resonance form reads them again (its lanes alone take 64 registers)
  constexpr bool KEEP = KB <= 8;
  __shared__ ddf s_red[(kBlock / 32) * NS > kBlock ? (kBlock / 32) * NS : kBlock];
  __shared__ unsigned s_bad[kBlock / 32];
  const int nbw = a.nbw;
  const double nr_re = a.has_nr ? a.cr[nbw] : 0.0, nr_im = a.has_nr ? a.ci[nbw] : 0.0;
  CohAcc<double, KB> acc;
  LogProduct lp;
#pragma unroll
  for (int k = 0; k < KA; ++k) acc.gre[k] = acc.gim[k] = 0.0;
  const int64_t n = a.n_total;
  for (int64_t i = begin + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < end;
       i += (int64_t)gridDim.x * blockDim.x) {
    double2 amp[KEEP ? KB : 1];
    if constexpr (KEEP) {
      // every load of the event before its first use (predicated, not a loop exit between them)
#pragma unroll
      for (int k = 0; k < KB; ++k) amp[k] = k < nbw ? cache[(int64_t)k * n + i] : make_double2(0.0, 0.0);
    }
    double sr = nr_re, si = nr_im;
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      if (k >= nbw) break;
      const double2 v = KEEP ? amp[k] : cache[(int64_t)k * n + i];
      sr = fma(a.cr[k], v.x, fma(-a.ci[k], v.y, sr));
      si = fma(a.cr[k], v.y, fma(a.ci[k], v.x, si));
    }
    const double s2 = fma(sr, sr, si * si);
    double inv;
    if (positive_normal(s2)) {
      lp.mul(s2);
      inv = rcp64(s2);
    } else if (s2 > 0.0) {  // subnormal or infinite
      acc.lf64 += log(s2);
      inv = 1.0 / s2;
    } else {
      acc.bad++;
      continue;
    }
    if constexpr (GRAD) {
      const double tr = sr * inv, ti = -si * inv;  // conj(S) / |S|^2
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        if (k >= nbw) break;
        const double2 v = KEEP ? amp[k] : cache[(int64_t)k * n + i];
        acc.gre[k] = fma(v.x, tr, fma(-v.y, ti, acc.gre[k]));
        acc.gim[k] = fma(v.x, ti, fma(v.y, tr, acc.gim[k]));
      }
      acc.gre[KB] += tr;  // A = 1
      acc.gim[KB] += ti;
    }
  }
  acc.lf64 += lp.log_value();
  coh_finish<double, KB, GRAD>(a, acc, begin, end, partials, counters, result, out_mode, s_red, s_bad);
}

// FP32 form with the amplitude-cache tiles staged in shared memory.  A tile holds
// kCohTile events of every float4 plane (aligned to multiples of kCohTile); bulk copies, one per
// plane, run kCohStages tiles ahead, the warps release the stages one by one (TileRing), and block b
// takes tiles tb0 + b, tb0 + b + gridDim.x, ...  Ragged first / last tiles are read from global
// memory.  Bound by HBM (64 bytes per event at 8 resonances; a plain read of 320 MB takes 48 us): 5M events
// 58.4 us (63.1 with a block barrier per tile).  Six stages were slower than four here as in a
// plain read (50 against 48 us).
// Dynamic shared memory: kCohStages * n_planes * kCohTile float4.
constexpr int kCohTile = kStagedBlock;  // one event per thread per tile
template <int KB>
constexpr int kCohStages = KB <= 8 ? 4 : 3;

template <int KB, bool GRAD>
__global__ void __launch_bounds__(kStagedBlock, 1) coh_nll_staged_kernel(const __grid_constant__ CohArgs<float> a,
                                                                   const float4* __restrict__ cache, int64_t begin,
                                                                   int64_t end, float2* partials, unsigned* counters,
                                                                   double* result, int out_mode) {
  constexpr int NS = CohLanes<float, KB, GRAD>::NS;
  constexpr int KA = KB + 1;
  constexpr int TE = kCohTile;
  constexpr int NST = kCohStages<KB>;
  constexpr int NP = (KB + 1) / 2;
  __shared__ ddf s_red[(kStagedBlock / 32) * NS > kStagedBlock ? (kStagedBlock / 32) * NS : kStagedBlock];
  __shared__ unsigned s_bad[kStagedBlock / 32];
  __shared__ __align__(8) TileRing<NST> s_ring;
  extern __shared__ __align__(128) float4 s_amp[];  // [NST][planes][TE]
  const int nbw = a.nbw;
  const int planes = (nbw + 1) / 2;
  const int64_t n = a.n_total;
  const int64_t tb0 = begin / TE, tb1 = (end + TE - 1) / TE;
  auto tile_of = [&](int j) { return tb0 + blockIdx.x + (int64_t)j * gridDim.x; };
  auto full = [&](int64_t t) { return t * TE >= begin && (t + 1) * TE <= end; };
  auto buf = [&](int st, int p) { return s_amp + ((size_t)st * planes + p) * TE; };
  grid_dep_wait();
  const unsigned withhold = withheld_tile(counters);  // the failure-detection test hook
  auto issue = [&](int j) {
    const int64_t t = tile_of(j);
    if (t >= tb1 || (withhold && j == (int)withhold - 1)) return;
    uint64_t* bar = &s_ring.bar[j % NST];
    s_ring.last[j % NST] = j;
    if (full(t)) {
      mbar_arrive_expect_tx(bar, (unsigned)(planes * TE * sizeof(float4)));
      for (int p = 0; p < planes; ++p) bulk_load(buf(j % NST, p), cache + (int64_t)p * n + t * TE, TE * sizeof(float4), bar);
    } else {
      mbar_arrive(bar);
    }
  };
  if (threadIdx.x == 0) {
    s_ring.init();
    for (int j = 0; j < NST; ++j) issue(j);
  }
  float2 cre[KA], cim[KA];
  {
    float cr[KA], ci[KA];
    coh_coeffs<float, KB>(a, cr, ci);
#pragma unroll
    for (int k = 0; k < KA; ++k) {
      cre[k] = pk::splat(cr[k]);
      cim[k] = pk::splat(ci[k]);
    }
  }
  Kahan lf;
  float2 G1[KA], G2[KA];
#pragma unroll
  for (int k = 0; k < KA; ++k) G1[k] = G2[k] = pk::splat(0.f);
  unsigned bad = 0;
  // absent planes stay zero: only the model's planes are loaded over these
  float4 v[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) v[p] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto event = [&]() {
    float2 amp[KB];
#pragma unroll
    for (int k = 0; k < KB; ++k) amp[k] = (k & 1) ? make_float2(v[k / 2].z, v[k / 2].w) : make_float2(v[k / 2].x, v[k / 2].y);
    coh_event_pk<KB, GRAD>(cre, cim, amp, lf, G1, G2, bad);
  };
  __syncthreads();  // barriers initialised before any thread waits on them
  const long long wlim = tile_wait_limit(counters);
  bool gave_up = false;
  for (int j = 0; tile_of(j) < tb1; ++j) {
    const int64_t t = tile_of(j);
    if (!s_ring.wait(j, wlim)) {
      gave_up = true;
      break;
    }
    if (full(t)) {
      const float4* sb = buf(j % NST, 0) + threadIdx.x;  // plane p of the event at sb[p * TE]
#pragma unroll
      for (int p = 0; p < NP; ++p)
        if (p < planes) v[p] = sb[p * TE];
      event();
    } else {
      const int64_t i = t * TE + threadIdx.x;
      if (i >= begin && i < end) {
#pragma unroll
        for (int p = 0; p < NP; ++p)
          if (p < planes) v[p] = __ldg(cache + (int64_t)p * n + i);
        event();
      }
    }
    s_ring.release(j, issue);
  }
  s_ring.finish(gave_up, counters);
  CohAcc<float, KB> acc;
  acc.lf32 = lf;
  acc.bad = bad;
#pragma unroll
  for (int k = 0; k < KA; ++k) {
    acc.gre[k] = G1[k].x - G2[k].y;
    acc.gim[k] = G1[k].y + G2[k].x;
  }
  coh_finish<float, KB, GRAD>(a, acc, begin, end, partials, counters, result, out_mode, s_red, s_bad);
}

// per-event log f = log|S|^2 - log N
template <typename T, int KB>
__global__ void coh_logf_kernel(const __grid_constant__ CohArgs<T> a, const void* cache_v, double logN,
                                double* __restrict__ out) {
  constexpr int KA = KB + 1;
  using Vec = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  const Vec* cache = (const Vec*)cache_v;
  const int nbw = a.nbw;
  const int64_t n = a.n_total;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    T ar[KA], ai[KA];
    load_amps<KB>(cache, n, i, nbw, ar, ai);
    ar[KB] = T(1);
    ai[KB] = T(0);
    T sr = T(0), si = T(0);
#pragma unroll
    for (int k = 0; k < KA; ++k) {
      const T c_r = k < nbw ? a.cr[k] : (k == KB && a.has_nr ? a.cr[nbw] : T(0));
      const T c_i = k < nbw ? a.ci[k] : (k == KB && a.has_nr ? a.ci[nbw] : T(0));
      sr += c_r * ar[k] - c_i * ai[k];
      si += c_r * ai[k] + c_i * ar[k];
    }
    const T s2 = sr * sr + si * si;
    out[i] = s2 > T(0) ? log((double)s2) - logN : -HUGE_VAL;
  }
}

// ---------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------
static double kallen(double a, double b, double c) { return a * a + b * b + c * c - 2 * a * b - 2 * a * c - 2 * b * c; }

static void pair_masses(const DalitzModel& d, int pair, double& mA, double& mB, double& mC) {
  if (pair == 0) {
    mA = d.m1;
    mB = d.m2;
    mC = d.m3;
  } else if (pair == 1) {
    mA = d.m1;
    mB = d.m3;
    mC = d.m2;
  } else {
    mA = d.m2;
    mB = d.m3;
    mC = d.m1;
  }
}

// Coefficient k of the amplitude sum from its two parameters: (Re, Im), or (r, phi) with
// GOO_COEF_POLAR.
static void coef(const DalitzModel& d, const double* theta, int k, double& re, double& im) {
  const double u = theta[d.par_re[k]], v = theta[d.par_im[k]];
  if (d.polar) {
    re = u * std::cos(v);
    im = u * std::sin(v);
  } else {
    re = u;
    im = v;
  }
}

// The polar Jacobian entries (cos phi, sin phi, r) of every amplitude into kernel arguments.
template <typename A>
static void fill_jacobian(const DalitzModel& d, const double* theta, A& a) {
  a.polar = d.polar ? 1 : 0;
  for (int k = 0; k < d.K; ++k) {
    a.jc[k] = d.polar ? std::cos(theta[d.par_im[k]]) : 1.0;
    a.js[k] = d.polar ? std::sin(theta[d.par_im[k]]) : 0.0;
    a.jr[k] = d.polar ? theta[d.par_re[k]] : 1.0;
  }
}

static uint64_t lineshape_key(const DalitzModel& d, const double* theta) {
  uint64_t h = 1469598103934665603ull;
  for (int k = 0; k < d.nbw; ++k) {
    double v[2] = {theta[d.par_m0[k]], theta[d.par_w[k]]};
    const unsigned char* p = (const unsigned char*)v;
    for (size_t j = 0; j < sizeof v; ++j) h = (h ^ p[j]) * 1099511628211ull;
  }
  return h ? h : 1;
}

// ---------------------------------------------------------------------------------------
// floating lineshapes (masses and widths free; paper Sec. 4: the cache is then invalid at
// every step).  No amplitude cache: each evaluation evaluates every Breit-Wigner amplitude of the
// events and of the MC sample from (s12, s13) with the
// parts of its denominator D = m0^2 - s - i m0 Gamma(s), which give
//   d log A / d m0     = rho - (2 m0 - i kappa m0 Gamma(s)) / D,
//   d log A / d Gamma0 = i m0 Gamma(s) / (Gamma0 D),
// where rho = d log(B_L(z) / B_L(z0)) / d m0 (through q0) and kappa = d log(m0 Gamma(s)) /
// d m0 = 2 / m0 - (2L + 1) d log q0 / d m0 + 2 rho are constants of the resonance (the
// spin and parent-barrier factors do not depend on m0 or Gamma0).  With u_k = A_k conj(S) w and
// y_k = c_k u_k / D_k (w = 1 / |S|^2 for events and 1 for MC points) the lanes are: 0 = sum log2 |S|^2
// (events) or sum |S|^2 (MC); per amplitude slot sum u_k (re, im); per resonance sum Re y_k and
// sum m0 Gamma(s) Im y_k.  The last block has
//   sum Re(c_k u_k d log A_k / d m0) = rho Re(c_k sum u_k) - 2 m0 sum Re y_k - kappa sum m0 Gamma Im y_k,
//   sum Re(c_k u_k d log A_k / d Gamma0) = -(sum m0 Gamma Im y_k) / Gamma0
// from both sets of sums and combines them:
//   NLL = -sum log |S|^2 + n log(sum_MC |S|^2 / n_MC),
//   d NLL / d p = -sum_events (d |S|^2 / d p) / |S|^2 + n (sum_MC d |S|^2 / d p) / sum_MC |S|^2.
//
// Issue-bound.  The factors shared by a pair and spin are formed once per point (lineshape.cuh) and kept
// in the thread's column of shared memory, and so are g_k = 1 / D_k and c_k g_k of every resonance for
// its lanes (A_k = h g_k with a real h, so u_k = h (g_k conj(S) w) and y_k = h (g_k conj(S) w) (c_k g_k)); FP32
// works on two points at a time; the first blocks of the one launch take the MC sample and the others the events, so that neither waits for the
// other's reduction.  5M events and 1M MC points, 8 resonances: 495 us in two launches with every
// resonance evaluated by itself, 144 us with the amplitudes formed a second time for the lanes, now
// 131 us in repeated calls and 137 us under ncu, a call 146 us (217 KB of shared memory; issue slots 57 %, FMA pipe 54 %,
// shared memory 53 % busy).
// ---------------------------------------------------------------------------------------
template <typename T>
struct LsConst {
  T cr[kMaxAmp], ci[kMaxAmp];          // coefficients by slot: resonances, then the NR in slot KB
  T nci[kMaxAmp];                      // -ci
  double rho[kMaxAmp], kappa[kMaxAmp], two_m0[kMaxAmp], inv_g0[kMaxAmp];
};

template <int KB, bool GRAD>
struct LsLanes {
  static constexpr int NS = GRAD ? 1 + 2 * (KB + 1) + 2 * KB : 1;
};

// One set of points (the MC sample or the events).
template <typename T>
struct LsSet {
  const T *c12, *c13;
  int64_t begin, end, n;  // the points of the evaluation, and of the column
};

// Threads per block: 16 warps per SM in one block (half as many partial sums for the last block as with two of
// 8), 8 where 15 resonances' lanes fill the register file.
template <int KB>
constexpr int kLsBlockOf = KB <= 8 ? kStagedBlock : kBlock;

// Dynamic shared memory: the shared factors of every thread, later the block reduction's lanes.
template <typename T, int KB, bool GRAD>
constexpr size_t ls_smem() {
  const size_t f = (size_t)(kLsCols + (GRAD ? 4 * KB : 0)) * kLsBlockOf<KB> * 8, r = (size_t)LsLanes<KB, GRAD>::NS * kLsBlockOf<KB> * sizeof(ddf);
  return f > r ? f : r;
}

namespace lsv {
// sums over a thread's points: a packed pair's two halves, or the double itself
__device__ __forceinline__ ddf total(float2 v) { return dd_add(ddf{v.x, 0.f}, ddf{v.y, 0.f}); }
__device__ __forceinline__ ddf total(double v) { return dd_from_double(v); }
}  // namespace lsv

// Compensated (FP32) or plain (FP64) running sum of lane 0.
struct LsSumF {
  Kahan a, b;
  __device__ __forceinline__ void add(float2 x) {
    a.add(x.x);
    b.add(x.y);
  }
  __device__ __forceinline__ ddf value() const { return dd_add(a.value(), b.value()); }
};
struct LsSumD {
  double s = 0.0;
  __device__ __forceinline__ void add(double x) { s += x; }
  __device__ __forceinline__ ddf value() const { return dd_from_double(s); }
};

// The point(s) of step j: (s12, s13), and which of them count.
__device__ __forceinline__ void ls_load(const LsSet<float>& D, int64_t j, float2& a, float2& b, bool& v0, bool& v1) {
  const int64_t i = 2 * j;  // pairs at even indices
  v0 = i >= D.begin;
  v1 = i + 1 < D.end;
  if (i + 1 < D.n) {
    a = *reinterpret_cast<const float2*>(D.c12 + i);
    b = *reinterpret_cast<const float2*>(D.c13 + i);
  } else {
    a = pk::splat(D.c12[i]);
    b = pk::splat(D.c13[i]);
  }
  if (!(v0 && v1)) {  // a point outside the range takes the other's place, with weight 0
    a = pk::splat(v0 ? a.x : a.y);
    b = pk::splat(v0 ? b.x : b.y);
  }
}
__device__ __forceinline__ void ls_load(const LsSet<double>& D, int64_t j, double& a, double& b, bool& v0, bool& v1) {
  a = D.c12[j];
  b = D.c13[j];
  v0 = true;
  v1 = false;
}
__device__ __forceinline__ int64_t ls_first(const LsSet<float>& D) { return D.begin >> 1; }
__device__ __forceinline__ int64_t ls_last(const LsSet<float>& D) { return (D.end + 1) >> 1; }
__device__ __forceinline__ int64_t ls_first(const LsSet<double>& D) { return D.begin; }
__device__ __forceinline__ int64_t ls_last(const LsSet<double>& D) { return D.end; }

// The weight 1 / |S|^2 (MC: 1) and lane 0's term (log2 |S|^2 in FP32, log in FP64; MC: |S|^2) of the points that
// count, 0 for the others; events with |S|^2 <= 0 are counted in bad.
__device__ __forceinline__ void ls_weight(bool mc, float2 s2, bool v0, bool v1, float2& w, float2& term, unsigned& bad) {
  if (mc) {
    w = make_float2(v0 ? 1.f : 0.f, v1 ? 1.f : 0.f);
    term = make_float2(v0 ? s2.x : 0.f, v1 ? s2.y : 0.f);
    return;
  }
  const bool ok0 = s2.x > 0.f, ok1 = s2.y > 0.f;
  bad += (unsigned)(v0 && !ok0) + (unsigned)(v1 && !ok1);
  float2 r, l;
  if (fminf(s2.x, s2.y) >= 1.17549435e-38f) {
    r = lsv::rcp(s2);
    l = make_float2(pk::lg2(s2.x), pk::lg2(s2.y));
  } else {  // the hardware functions take a subnormal number for 0
    r = make_float2(1.f / s2.x, 1.f / s2.y);
    l = make_float2(log2f(s2.x), log2f(s2.y));
  }
  w = make_float2(v0 && ok0 ? r.x : 0.f, v1 && ok1 ? r.y : 0.f);
  term = make_float2(v0 && ok0 ? l.x : 0.f, v1 && ok1 ? l.y : 0.f);
}
__device__ __forceinline__ void ls_weight(bool mc, double s2, bool, bool, double& w, double& term, unsigned& bad) {
  if (mc) {
    w = 1.0;
    term = s2;
  } else if (s2 > 0.0) {
    w = recip(s2);
    term = log(s2);
  } else {
    ++bad;
    w = term = 0.0;
  }
}

template <typename T, int KB, bool GRAD>
__global__ void __launch_bounds__(kLsBlockOf<KB>, 1)
    coh_ls_kernel(const __grid_constant__ CohArgs<T> a, const __grid_constant__ LsConst<T> c,
                  const __grid_constant__ LsTables<T> t, const __grid_constant__ LsSet<T> mc,
                  const __grid_constant__ LsSet<T> ev, int nb_mc, float2* partials, unsigned* counters, double* out,
                  int out_mode) {
  using namespace lsv;
  using V = typename std::conditional<sizeof(T) == 4, float2, double>::type;
  using Sum = typename std::conditional<sizeof(T) == 4, LsSumF, LsSumD>::type;
  constexpr int KA = KB + 1;
  constexpr int NT = kLsBlockOf<KB>;
  constexpr int NS = LsLanes<KB, GRAD>::NS;
  __shared__ ddf s_red[NT / 32];
  __shared__ double s_out[NS], s_mc[NS];
  extern __shared__ __align__(16) unsigned char s_dyn[];
  V* s_v = reinterpret_cast<V*>(s_dyn);
  V *sc = s_v + threadIdx.x, *gc = sc + 3 * NT, *hc = sc + 12 * NT, *ac = sc + kLsCols * NT;
  const bool is_mc = (int)blockIdx.x < nb_mc;
  const LsSet<T>& D = is_mc ? mc : ev;
  const int nb = is_mc ? nb_mc : (int)gridDim.x - nb_mc, b0 = is_mc ? (int)blockIdx.x : (int)blockIdx.x - nb_mc;
  Sum l0;
  V lre[KA], lim[KA], lwr[KB], lwi[KB];
  const V zero = splat(V{}, T(0));
#pragma unroll
  for (int k = 0; k < KA; ++k) lre[k] = lim[k] = zero;
#pragma unroll
  for (int k = 0; k < KB; ++k) lwr[k] = lwi[k] = zero;
  unsigned bad = 0;
  const int64_t last = ls_last(D);
  for (int64_t j = ls_first(D) + b0 * (int64_t)NT + threadIdx.x; j < last; j += (int64_t)nb * NT) {
    V x12, x13;
    bool v0, v1;
    ls_load(D, j, x12, x13, v0, v1);
    ls_groups<T, V>(t, x12, x13, sc, gc, hc, NT);
    V sr = splat(V{}, c.cr[KB]), si = splat(V{}, c.ci[KB]);  // the non-resonant amplitude is 1
#pragma unroll 4
    for (int k = 0; k < t.nbw; ++k) {
      // g = 1 / D, A_k = h g with a real h; c_k g serves the sum and the mass and width lanes
      V gr, gi, di;
      ls_propagator<T, V>(t, k, sc, gc, NT, gr, gi, di);
      const V h = ls_numerator<T, V>(t, k, hc, NT), cr = splat(V{}, c.cr[k]);
      const V qr = fma(cr, gr, mul(splat(V{}, c.nci[k]), gi)), qi = fma(cr, gi, mul(splat(V{}, c.ci[k]), gr));
      sr = fma(h, qr, sr);
      si = fma(h, qi, si);
      if constexpr (GRAD) {
        ac[4 * k * NT] = gr;
        ac[(4 * k + 1) * NT] = gi;
        ac[(4 * k + 2) * NT] = qr;
        ac[(4 * k + 3) * NT] = qi;
      }
    }
    V w, term;
    ls_weight(is_mc, fma(sr, sr, mul(si, si)), v0, v1, w, term, bad);
    l0.add(term);
    if constexpr (GRAD) {
      const V tr = mul(sr, w), mti = mul(si, w), ti = neg(mti);  // conj(S) w
      lre[KB] = add(lre[KB], tr);  // the non-resonant slot: A = 1
      lim[KB] = add(lim[KB], ti);
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        if (k >= t.nbw) break;
        const V gr = ac[4 * k * NT], gi = ac[(4 * k + 1) * NT], qr = ac[(4 * k + 2) * NT], qi = ac[(4 * k + 3) * NT];
        const V h = ls_numerator<T, V>(t, k, hc, NT);
        const V ur = fma(gr, tr, mul(gi, mti)), ui = fma(gr, ti, mul(gi, tr));  // conj(S) w / D_k
        lre[k] = fma(h, ur, lre[k]);
        lim[k] = fma(h, ui, lim[k]);
        // y_k = c_k A_k conj(S) w / D_k
        lwr[k] = fma(h, sub(mul(ur, qr), mul(ui, qi)), lwr[k]);
        lwi[k] = fma(mul(h, ls_width<T, V>(t, k, gc, NT)), fma(ur, qi, mul(ui, qr)), lwi[k]);
      }
    }
  }
  ddf v[NS];
  v[0] = l0.value();
  if (sizeof(T) == 4 && !is_mc) v[0] = dd_mul(v[0], ddf{kLn2Hi, kLn2Lo});
  if constexpr (GRAD) {
#pragma unroll
    for (int k = 0; k < KA; ++k) {
      v[1 + 2 * k] = total(lre[k]);
      v[2 + 2 * k] = total(lim[k]);
    }
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      v[1 + 2 * KA + 2 * k] = total(lwr[k]);
      v[2 + 2 * KA + 2 * k] = total(lwi[k]);
    }
  }
  for (int m = 16; m > 0; m >>= 1) bad += __shfl_xor_sync(0xffffffffu, bad, m);
  if ((threadIdx.x & 31) == 0 && bad) atomicAdd(counters + 1, bad);
  __syncthreads();  // the columns of the shared factors become the reduction's buffer
  block_reduce_transpose<NS>(v, partials, reinterpret_cast<ddf*>(s_dyn));
  if (!last_block_ticket(counters, gridDim.x)) return;
  unsigned nbad = 0u, status = 0u;
  if (threadIdx.x == 0) {
    nbad = __ldcg(counters + 1);
    status = __ldcg(counters + kStatusWord);
  }
  reduce_partials<24>(partials, NS, nb_mc, s_mc, s_red, NT);
  reduce_partials<24>(partials + (size_t)nb_mc * NS, NS, (int)gridDim.x - nb_mc, s_out, s_red, NT);
  const double nev = (double)(ev.end - ev.begin), Smc = s_mc[0];
  const int P = a.n_params;
  const int off = out_mode == 0 ? 2 : 3;
  if constexpr (GRAD) {
    __shared__ double s_term[4 * kMaxAmp];
    const double f = nev / Smc;
    // -2 (events) + 2 n / S_mc (MC) of lane j
    auto both = [&](int j) { return 2.0 * fma(f, s_mc[j], -s_out[j]); };
    if ((int)threadIdx.x < a.K) {
      const int k = threadIdx.x, sl = k < a.nbw ? k : KB;  // the NR lives in the last slot
      double gre = both(1 + 2 * sl), gim = -both(2 + 2 * sl);
      coef_chain(a.polar, a.jc[k], a.js[k], a.jr[k], gre, gim);
      s_term[2 * k] = gre;
      s_term[2 * k + 1] = gim;
    } else if (threadIdx.x >= 32 && (int)threadIdx.x < 32 + a.nbw) {
      const int k = threadIdx.x - 32;
      const double cu = (double)c.cr[k] * both(1 + 2 * k) - (double)c.ci[k] * both(2 + 2 * k);
      const double y = both(2 + 2 * KA + 2 * k);
      s_term[2 * (a.K + k)] = c.rho[k] * cu - c.two_m0[k] * both(1 + 2 * KA + 2 * k) - c.kappa[k] * y;
      s_term[2 * (a.K + k) + 1] = -c.inv_g0[k] * y;
    }
    __syncthreads();
    for (int p = threadIdx.x; p < P; p += blockDim.x) out[off + p] = a.map.gather(p, s_term);
  } else {
    for (int p = threadIdx.x; p < P; p += blockDim.x) out[off + p] = 0.0;
  }
  if (threadIdx.x == 0) {
    counters[1] = 0u;
    counters[kStatusWord] = 0u;
    *counters = 0u;  // the ticket
    const double N = Smc / (double)(mc.end - mc.begin);
    const double nb_ = status ? -1.0 : (double)nbad;  // a device wait that gave up: negative count
    out[0] = -s_out[0] + nev * log(N);
    if (out_mode == 0) {
      out[1] = nb_;
      out[2 + P] = N;
    } else {
      out[1] = 0.0;
      out[2] = nb_;
    }
  }
  result_complete(out);
}

// ---------------------------------------------------------------------------------------
// time-dependent three-body model (GOO_OP_TD3; paper Sec. 5, Table 2).  The anti-particle's
// amplitudes are the same lineshapes at the exchanged point, abar_k(s12, s13) =
// a_k(s13, s12) (a second cache built from the exchanged columns); A = sum c_k a_k,
// B = sum c_k abar_k with the same coefficients.  Per event the four decay-time terms of the
// four-body model (timeterms.cuh) give
//   R = (|A|^2+|B|^2)/2 T_ch + (|A|^2-|B|^2)/2 T_c + Re(AB*) T_sh + Im(AB*) T_s,
// and the gradient lanes Re / -Im of (a_k V_A + abar_k V_B) / R with
//   V_A = (T_ch + T_c) A* + (T_sh - i T_s) B*,  V_B = (T_ch - T_c) B* + (T_sh + i T_s) A*,
// plus the four decay-time lanes of timeterms.cuh.  N comes from three MC Gram matrices,
//   <|A|^2> = c^T G_aa c*, <|B|^2> = c^T G_bb c*, <AB*> = c^T G_ab c*,
// and the closed-form time integrals.
// ---------------------------------------------------------------------------------------

constexpr int kTd3KB = 15;  // resonance slots of the time-dependent three-body kernels (NR in slot 15)

template <typename T>
struct Td3Args {
  T cr[kTd3KB + 1], ci[kTd3KB + 1];  // coefficients by slot: resonances, then the NR in slot kTd3KB
  T G, x, y, s;                      // 1/tau, mixing, resolution in the path's precision
  TimeCoef<T> tc;                    // the same with the moment-series coefficients
  T wa[kWMax];                       // Weideman coefficients
  T wL;
  int wN, nbw, K, n_params;
  // terms 2k, 2k + 1: the coefficient parameters of amplitude k (tree order); 2 kMaxAmp + j: the time
  // parameters
  GradMap<2 * kMaxAmp + 4> map;
  int64_t n_total;                   // events of the dataset (cache plane length)
  int polar;                         // the coefficient parameters are (r, phi)
  double jc[kMaxAmp], js[kMaxAmp], jr[kMaxAmp];  // cos phi, sin phi, r per amplitude (polar)
  // the normalisation at theta, formed on the host in FP64 from the cached Gram matrices
  // (td3_norm_terms): N, log N, (dN / d Re c_k) / N, (dN / d Im c_k) / N (tree order) and
  // (dN / dx) / N, (dN / dy) / N, (tau dN / d tau) / N
  double nrm_N, nrm_logN, nrm_re[kMaxAmp], nrm_im[kMaxAmp], nrm_dt[3];
};

template <bool GRAD>
struct Td3Lanes {
  static constexpr int NS = GRAD ? 1 + 2 * (kTd3KB + 1) + 4 : 1;
};

// Block and last-block reductions of the lanes and the FP64 combination with the normalisation
// terms the host formed from the three Gram matrices (they depend on theta and the MC sample
// only).  lf: the thread's sum of log R as a double-float.
template <typename T, bool GRAD>
__device__ __forceinline__ void td3_finish(const Td3Args<T>& a, ddf lf, const T (&lre)[kTd3KB + 1],
                                           const T (&lim)[kTd3KB + 1], const T (&lt)[4], unsigned bad, int64_t begin,
                                           int64_t end, float2* partials, unsigned* counters, double* out, int out_mode,
                                           ddf* s_red, unsigned* s_bad) {
  constexpr int KB = kTd3KB, KA = KB + 1;
  constexpr int NS = Td3Lanes<GRAD>::NS;
  __shared__ double s_out[NS];
  const int nbw = a.nbw;
  ddf v[NS];
  v[0] = lf;
  if constexpr (GRAD) {
#pragma unroll
    for (int k = 0; k < KA; ++k) {
      v[1 + 2 * k] = (sizeof(T) == 4) ? ddf{(float)lre[k], 0.f} : dd_from_double((double)lre[k]);
      v[2 + 2 * k] = (sizeof(T) == 4) ? ddf{(float)lim[k], 0.f} : dd_from_double((double)lim[k]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
      v[1 + 2 * KA + j] = (sizeof(T) == 4) ? ddf{(float)lt[j], 0.f} : dd_from_double((double)lt[j]);
  }
  for (int m = 16; m > 0; m >>= 1) bad += __shfl_xor_sync(0xffffffffu, bad, m);
  if ((threadIdx.x & 31) == 0) s_bad[threadIdx.x >> 5] = bad;
  block_reduce_to_partials<NS>(v, NS, partials, s_red);
  if (threadIdx.x == 0) {
    unsigned b = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) b += s_bad[w];
    if (b) atomicAdd(counters + 1, b);
  }
  if (!last_block_ticket(counters, gridDim.x)) return;
  // Every other block added to the counter words before its ticket (and a fence): plain L2
  // reads, issued before the reduction so that their latency overlaps it.
  unsigned nbad = 0u, status = 0u;
  if (threadIdx.x == 0) {
    nbad = __ldcg(counters + 1);
    status = __ldcg(counters + kStatusWord);
  }
  reduce_partials(partials, NS, gridDim.x, s_out, s_red, blockDim.x);
  const int K = a.K;
  const double nev = (double)(end - begin);
  const int P = a.n_params;
  const int off = out_mode == 0 ? 2 : 3;
  if constexpr (GRAD) {
    __shared__ double s_term[2 * kMaxAmp + 4];
    if ((int)threadIdx.x < K) {
      const int k = threadIdx.x, sl = k < nbw ? k : KB;
      double gre = fma(nev, a.nrm_re[k], -s_out[1 + 2 * sl]), gim = fma(nev, a.nrm_im[k], -s_out[2 + 2 * sl]);
      coef_chain(a.polar, a.jc[k], a.js[k], a.jr[k], gre, gim);
      s_term[2 * k] = gre;
      s_term[2 * k + 1] = gim;
    } else if (threadIdx.x >= 32 && threadIdx.x < 36) {
      const int j = threadIdx.x - 32;
      s_term[2 * kMaxAmp + j] = (j < 3 ? nev * a.nrm_dt[j] : 0.0) -
                                time_gradient(j, (double)a.G, (double)a.x, (double)a.y, (double)a.s, s_out + 1 + 2 * KA, nev);
    }
    __syncthreads();
    for (int p = threadIdx.x; p < P; p += blockDim.x) out[off + p] = a.map.gather(p, s_term);
  } else {
    for (int p = threadIdx.x; p < P; p += blockDim.x) out[off + p] = 0.0;
  }
  if (threadIdx.x == 0) {
    counters[1] = 0u;
    counters[kStatusWord] = 0u;
    *counters = 0u;  // the ticket
    const double nb = status ? -1.0 : (double)nbad;  // a device wait that gave up: negative count
    out[0] = -s_out[0] + nev * a.nrm_logN;
    if (out_mode == 0) {
      out[1] = nb;
      out[2 + P] = a.nrm_N;
    } else {
      out[1] = 0.0;
      out[2] = nb;
    }
  }
  result_complete(out);
}

// FP32: all amplitude planes of the event are requested before any is used (loads
// predicated on the plane count rather than a loop exit, so none waits on the arithmetic of
// the one before), and kept for the gradient lanes; the sums run as packed (re, im) FMAs on the
// planes' halves, (sum cr_k a_k) and (sum ci_k a_k) per cache, combined once: four packed FMAs per
// amplitude, not eight.
template <bool GRAD>
__global__ void __launch_bounds__(kBlock, 2)
    td3_nll_f32_kernel(const __grid_constant__ Td3Args<float> a, const float4* __restrict__ cache_a,
                       const float4* __restrict__ cache_b, const float* __restrict__ tcol, int64_t begin, int64_t end,
                       float2* partials, unsigned* counters, double* out, int out_mode) {
  using namespace pk;
  constexpr int KB = kTd3KB, KA = KB + 1;
  constexpr int NS = Td3Lanes<GRAD>::NS;
  __shared__ ddf s_red[(kBlock / 32) * NS > kBlock ? (kBlock / 32) * NS : kBlock];
  __shared__ unsigned s_bad[kBlock / 32];
  const int64_t n = a.n_total;
  const int nbw = a.nbw;
  constexpr int NP = (KB + 1) / 2;
  float4 pa[NP], pb[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) pa[q] = pb[q] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto amp_a = [&](int k) { return (k & 1) ? make_float2(pa[k / 2].z, pa[k / 2].w) : make_float2(pa[k / 2].x, pa[k / 2].y); };
  auto amp_b = [&](int k) { return (k & 1) ? make_float2(pb[k / 2].z, pb[k / 2].w) : make_float2(pb[k / 2].x, pb[k / 2].y); };
  Kahan lf32;
  float lre[KA], lim[KA], lt[4];
#pragma unroll
  for (int k = 0; k < KA; ++k) lre[k] = lim[k] = 0.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) lt[j] = 0.f;
  unsigned bad = 0;
  for (int64_t i = begin + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < end;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float t = tcol[i];
#pragma unroll
    for (int q = 0; q < NP; ++q)
      if (2 * q < nbw) {
        pa[q] = __ldg(cache_a + (int64_t)q * n + i);
        pb[q] = __ldg(cache_b + (int64_t)q * n + i);
      }
    // the NR amplitude is 1 for both
    float2 P1 = make_float2(a.cr[KB], a.ci[KB]), P2 = splat(0.f), Q1 = P1, Q2 = splat(0.f);
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      if (k >= nbw) break;
      const float2 ak = amp_a(k), bk = amp_b(k);
      P1 = fma(splat(a.cr[k]), ak, P1);
      P2 = fma(splat(a.ci[k]), ak, P2);
      Q1 = fma(splat(a.cr[k]), bk, Q1);
      Q2 = fma(splat(a.ci[k]), bk, Q2);
    }
    const float Ar = P1.x - P2.y, Ai = P1.y + P2.x, Br = Q1.x - Q2.y, Bi = Q1.y + Q2.x;
    TimeTerms<float> tt;
    time_terms_g<float>(TdMath<float>{}, a.tc, a.wa, a.wN, a.wL, t, tt);
    const float AA = fma_rn(Ar, Ar, mul_rn(Ai, Ai)), BB = fma_rn(Br, Br, mul_rn(Bi, Bi));
    const float ABr = fma_rn(Ar, Br, mul_rn(Ai, Bi)), ABi = fma_rn(Ai, Br, -mul_rn(Ar, Bi));  // A conj(B)
    const float R = td_rate(tt, AA, BB, ABr, ABi);
    if (!(R > 0.f)) {
      ++bad;
      continue;
    }
    lf32.add(lg2(R));  // log2 R, scaled by ln 2 at the end
    if constexpr (GRAD) {
      const float invR = rcp(R);
      const float cp = 2.f * tt.P * invR, cm = 2.f * tt.Q * invR, sh = tt.Tsh * invR, ss = tt.Ts * invR;
      // V_A / R = cp A* + (sh - i ss) B*,  V_B / R = cm B* + (sh + i ss) A*
      const float VAr = cp * Ar + sh * Br - ss * Bi, VAi = -cp * Ai - sh * Bi - ss * Br;
      const float VBr = cm * Br + sh * Ar + ss * Ai, VBi = -cm * Bi - sh * Ai + ss * Ar;
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        if (k >= nbw) break;
        const float2 ak = amp_a(k), bk = amp_b(k);
        const float qr = ak.x * VAr - ak.y * VAi + bk.x * VBr - bk.y * VBi;  // Re(a V_A + abar V_B) / R
        const float qi = ak.x * VAi + ak.y * VAr + bk.x * VBi + bk.y * VBr;
        lre[k] += qr;
        lim[k] -= qi;
      }
      lre[KB] += VAr + VBr;  // the NR slot (a = abar = 1)
      lim[KB] -= VAi + VBi;
      time_lanes(a.tc, t, tt, AA, BB, ABr, ABi, invR, lt);
    }
  }
  td3_finish<float, GRAD>(a, dd_mul(lf32.value(), ddf{kLn2Hi, kLn2Lo}), lre, lim, lt, bad, begin, end, partials, counters,
                          out, out_mode, s_red, s_bad);
}

// FP64: bound by the FP64 pipe's slots (fp64.cuh), as the four-body kernel: FMA chains, exp and
// erfcx from tables in shared memory, the logarithm as a running product, tests on the integer
// pipe, the amplitudes read again for the gradient lanes.  0.4M events with the gradient: 751 -> 369 us
// per call (with the derivatives' closed form of timeterms.cuh).
template <bool GRAD>
__global__ void __launch_bounds__(kBlock, 2)
    td3_nll_f64_kernel(const __grid_constant__ Td3Args<double> a, const double2* __restrict__ cache_a,
                       const double2* __restrict__ cache_b, const double* __restrict__ tcol,
                       const Fp64Tables* __restrict__ tables, int64_t begin, int64_t end, float2* partials,
                       unsigned* counters, double* out, int out_mode) {
  constexpr int KB = kTd3KB, KA = KB + 1;
  constexpr int NS = Td3Lanes<GRAD>::NS;
  __shared__ ddf s_red[(kBlock / 32) * NS > kBlock ? (kBlock / 32) * NS : kBlock];
  __shared__ unsigned s_bad[kBlock / 32];
  __shared__ TimeTables s_tab;
  load_fp64_tables(s_tab, tables);
  const TdMath<double> F{s_tab};
  const int64_t n = a.n_total;
  const int nbw = a.nbw;
  LogProduct lp;
  double lf64 = 0.0;
  double lre[KA], lim[KA], lt[4];
#pragma unroll
  for (int k = 0; k < KA; ++k) lre[k] = lim[k] = 0.0;
#pragma unroll
  for (int j = 0; j < 4; ++j) lt[j] = 0.0;
  unsigned bad = 0;
  __syncthreads();
  for (int64_t i = begin + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < end;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double t = tcol[i];
    double Ar = a.cr[KB], Ai = a.ci[KB], Br = a.cr[KB], Bi = a.ci[KB];  // the NR amplitude is 1 for both
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      if (k >= nbw) break;
      const double2 va = __ldg(cache_a + (int64_t)k * n + i), vb = __ldg(cache_b + (int64_t)k * n + i);
      Ar = fma(a.cr[k], va.x, fma(-a.ci[k], va.y, Ar));
      Ai = fma(a.cr[k], va.y, fma(a.ci[k], va.x, Ai));
      Br = fma(a.cr[k], vb.x, fma(-a.ci[k], vb.y, Br));
      Bi = fma(a.cr[k], vb.y, fma(a.ci[k], vb.x, Bi));
    }
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
      ++bad;
      continue;
    }
    if constexpr (GRAD) {
      const double cp = 2.0 * tt.P * invR, cm = 2.0 * tt.Q * invR, sh = tt.Tsh * invR, ss = tt.Ts * invR;
      // V_A / R = cp A* + (sh - i ss) B*,  V_B / R = cm B* + (sh + i ss) A*; m...i: minus the imaginary part
      const double VAr = fma(cp, Ar, fma(sh, Br, -ss * Bi)), mVAi = fma(cp, Ai, fma(sh, Bi, ss * Br));
      const double VBr = fma(cm, Br, fma(sh, Ar, ss * Ai)), mVBi = fma(cm, Bi, fma(sh, Ai, -ss * Ar));
#pragma unroll
      for (int k = 0; k < KB; ++k) {
        if (k >= nbw) break;
        const double2 va = __ldg(cache_a + (int64_t)k * n + i), vb = __ldg(cache_b + (int64_t)k * n + i);
        lre[k] = fma(va.x, VAr, fma(va.y, mVAi, fma(vb.x, VBr, fma(vb.y, mVBi, lre[k]))));
        lim[k] = fma(va.x, mVAi, fma(-va.y, VAr, fma(vb.x, mVBi, fma(-vb.y, VBr, lim[k]))));
      }
      lre[KB] += VAr + VBr;  // the NR slot (a = abar = 1)
      lim[KB] += mVAi + mVBi;
      time_lanes(a.tc, t, tt, AA, BB, ABr, ABi, invR, lt);
    }
  }
  lf64 += lp.log_value();
  td3_finish<double, GRAD>(a, dd_from_double(lf64), lre, lim, lt, bad, begin, end, partials, counters, out, out_mode,
                           s_red, s_bad);
}

// The tables of lineshape.cuh from the per-resonance constants of `d.host` (FP64, rounded once).
template <typename T>
static void fill_ls_tables(const DalitzModel& d, LsTables<T>& t) {
  std::memset(&t, 0, sizeof t);
  const DalitzDev& h = d.host;
  t.sum_hi = (T)h.sumsq;
  t.sum_lo = (T)(h.sumsq - (double)t.sum_hi);
  t.r2 = (T)(d.r_res * d.r_res);
  t.zpk = (T)(d.r_par * d.r_par / (4 * d.M * d.M));
  t.nbw = d.nbw;
  for (int k = 0; k < d.nbw; ++k) {
    const BwConst& b = h.bw[k];
    typename LsTables<T>::Pair& P = t.pair[b.pair];
    P.thrP = (T)b.thrP;
    P.thrM = (T)b.thrM;
    P.pthrP = (T)b.pthrP;
    P.pthrM = (T)b.pthrM;
    P.zconst = (T)b.zconst;
    typename LsTables<T>::Res& R = t.res[k];
    R.m0sq = (T)b.m0sq;
    R.c1 = (T)(b.m0w * b.m0 * b.Fz0 * std::pow(b.inv_q0sq, b.spin + 0.5));
    R.c2 = (T)std::sqrt(b.Fz0);
    R.group = 3 * b.pair + b.spin;
    t.groups |= 1 << R.group;
  }
}

// Lineshape constants for the current theta (FP64, once per lineshape version).
static int dalitz_constants(goo_model* m, const double* theta) {
  DalitzModel& d = *m->dalitz;
  const uint64_t key = lineshape_key(d, theta);
  if (key == d.ls_key) return GOO_OK;
  DalitzDev& h = d.host;
  h.nbw = d.nbw;
  const double M = d.M;
  h.sumsq = M * M + d.m1 * d.m1 + d.m2 * d.m2 + d.m3 * d.m3;
  for (int k = 0; k < d.nbw; ++k) {
    BwConst& b = h.bw[k];
    const int L = d.spin[k];
    double mA, mB, mC;
    pair_masses(d, d.pair[k], mA, mB, mC);
    const double m0 = theta[d.par_m0[k]], g0 = theta[d.par_w[k]];
    if (!(m0 > mA + mB) || !(g0 > 0))
      return set_error(GOO_ERR_ARG, "amplitude %d: mass %g must exceed its threshold %g and width %g be > 0", k, m0,
                       mA + mB, g0);
    b.spin = L;
    b.pair = d.pair[k];
    b.m0sq = m0 * m0;
    b.m0w = m0 * g0;
    const double q0sq = kallen(m0 * m0, mA * mA, mB * mB) / (4 * m0 * m0);
    b.inv_q0sq = 1.0 / q0sq;
    b.r2 = d.r_res * d.r_res;
    b.rp2 = d.r_par * d.r_par;
    b.thrP = (mA + mB) * (mA + mB);
    b.thrM = (mA - mB) * (mA - mB);
    b.pthrP = (M + mC) * (M + mC);
    b.pthrM = (M - mC) * (M - mC);
    b.zconst = (mA * mA - mB * mB) * (M * M - mC * mC);
    b.inv4M2 = 1.0 / (4 * M * M);
    const double z0 = b.r2 * q0sq;
    b.Fz0 = (L == 1) ? 1.0 + z0 : (L == 2 ? 9.0 + 3.0 * z0 + z0 * z0 : 1.0);
    b.m0 = m0;
    BwConstT<float>& f = h.bwf[k];
    f.spin = b.spin;
    f.pair = b.pair;
    f.m0sq = (float)b.m0sq;
    f.m0w = (float)b.m0w;
    f.inv_q0sq = (float)b.inv_q0sq;
    f.r2 = (float)b.r2;
    f.rp2 = (float)b.rp2;
    f.thrP = (float)b.thrP;
    f.thrM = (float)b.thrM;
    f.pthrP = (float)b.pthrP;
    f.pthrM = (float)b.pthrM;
    f.zconst = (float)b.zconst;
    f.inv4M2 = (float)b.inv4M2;
    f.Fz0 = (float)b.Fz0;
    f.m0 = (float)b.m0;
  }
  fill_ls_tables(d, d.ls64);
  fill_ls_tables(d, d.ls32);
  d.ls_key = key;
  d.gram_key[0] = d.gram_key[1] = 0;
  d.gram3_key[0] = d.gram3_key[1] = 0;
  return GOO_OK;
}

// The device copy of the per-resonance constants (the toy generator's) at the current
// lineshapes.
static int dalitz_dev(goo_model* m) {
  DalitzModel& d = *m->dalitz;
  if (d.dev_key == d.ls_key) return GOO_OK;
  GOO_CUDA_TRY(cudaMemcpyAsync(d.dev, &d.host, sizeof(DalitzDev), cudaMemcpyHostToDevice, m->ctx->stream));
  GOO_CUDA_TRY(cudaStreamSynchronize(m->ctx->stream));
  d.dev_key = d.ls_key;
  return GOO_OK;
}

// Builds (if stale) the amplitude cache of `ds` in `precision`; returns its device pointer.
// With `exchanged`, the amplitudes at the exchanged Dalitz point (s13, s12): the anti-particle
// amplitudes of the time-dependent three-body model.
// behind_gram: the kernel before it in the stream is a Gram kernel (of other caches).
static int ensure_cache(goo_model* m, const goo_dataset* ds_c, int precision, const void** out,
                        bool exchanged = false, bool behind_gram = false) {
  goo_dataset* ds = const_cast<goo_dataset*>(ds_c);
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  const int pi = precision == GOO_F32 ? 0 : 1;
  const uint64_t key = d.ls_key ^ (uint64_t)(uintptr_t)m ^ (uint64_t)(pi + 1 + (exchanged ? 4 : 0)) * 0x9e3779b97f4a7c15ull ^
                       ds->epoch * 0xd6e8feb86659fd93ull;
  CacheSlot& slot = ds->cache[pi + (exchanged ? 2 : 0)];
  const int ca = exchanged ? d.col13 : d.col12, cb = exchanged ? d.col12 : d.col13;
  const int64_t n = ds->n;
  const size_t bytes = pi == 0 ? (size_t)((d.nbw + 1) / 2) * (size_t)n * sizeof(float4)
                               : (size_t)d.nbw * (size_t)n * sizeof(double2);
  if (slot.ptr && slot.key == key && slot.bytes >= bytes) {
    *out = slot.ptr;
    return GOO_OK;
  }
  if (!slot.ptr || slot.bytes < bytes) {
    if (slot.ptr) cudaFree(slot.ptr);
    slot.ptr = nullptr;
    slot.bytes = 0;
    if (cudaMalloc(&slot.ptr, bytes > 0 ? bytes : 16) != cudaSuccess) {
      cudaGetLastError();
      return set_error(GOO_ERR_OOM, "amplitude cache of %zu bytes does not fit", bytes);
    }
    slot.bytes = bytes;
  }
  if (n > 0 && d.nbw > 0) {
    const void* fn = pi == 0 ? (const void*)amp_cache_f32_kernel : (const void*)amp_cache_f64_kernel;
    const int64_t need = ((pi == 0 ? (n + 1) / 2 : n) + kLsBlock - 1) / kLsBlock;
    const int nb = (int)std::min<int64_t>(need, (int64_t)ctx->num_sms * cached_occupancy(fn, ctx->device, kLsBlock, 0));
    LaunchScope ls(ctx, pi == 0 ? "amp_cache_f32" : "amp_cache_f64");
    if (pi == 0 && behind_gram)
      GOO_CUDA_TRY(launch_early(amp_cache_f32_kernel, nb, kLsBlock, 0, ctx->stream, d.ls32, ds->d32[ca], ds->d32[cb], n,
                                (float4*)slot.ptr));
    else if (pi == 0)
      amp_cache_f32_kernel<<<nb, kLsBlock, 0, ctx->stream>>>(d.ls32, ds->d32[ca], ds->d32[cb], n, (float4*)slot.ptr);
    else if (behind_gram)
      GOO_CUDA_TRY(launch_early(amp_cache_f64_kernel, nb, kLsBlock, 0, ctx->stream, d.ls64, ds->d64[ca], ds->d64[cb], n,
                                (double2*)slot.ptr));
    else
      amp_cache_f64_kernel<<<nb, kLsBlock, 0, ctx->stream>>>(d.ls64, ds->d64[ca], ds->d64[cb], n, (double2*)slot.ptr);
    GOO_CUDA_TRY(cudaGetLastError());
  }
  slot.key = key;
  *out = slot.ptr;
  return GOO_OK;
}

// The Gram matrix at the current lineshapes.  `ds`: a dataset whose cache the caller needs next; when the
// matrix is rebuilt, so is that cache, behind the Gram kernel, and the GPU is busy while the host takes the
// matrix and launches the likelihood; the three launches overlap at their ends (launch_early).  2M events,
// 1M MC points: 123 us a point one after the other, 119 us queued behind, 108 us overlapped.
static int ensure_gram(goo_model* m, int precision, const goo_dataset* ds = nullptr) {
  DalitzModel& d = *m->dalitz;
  const int pi = precision == GOO_F32 ? 0 : 1;
  if (!d.mc) return set_error(GOO_ERR_STATE, "amplitude model has no MC normalisation sample (goo_model_set_norm)");
  const uint64_t key = d.ls_key ^ (uint64_t)(uintptr_t)d.mc ^ (uint64_t)(pi + 7) ^ d.mc->epoch * 0xd6e8feb86659fd93ull;
  if (d.gram_key[pi] == key) return GOO_OK;
  const void* cache = nullptr;
  GOO_TRY(ensure_cache(m, d.mc, precision, &cache));
  if (d.mc->n < 1) return set_error(GOO_ERR_ARG, "the MC normalisation sample is empty");
  GOO_TRY(gram_matrices(m->ctx, precision, false, 1, &cache, &cache, d.mc->n, d.nbw, d.K, d.gram_host[pi],
                        pi == 0 ? "gram_f32" : "gram_f64", [&]() -> int {
                          const void* c = nullptr;
                          return ds ? ensure_cache(m, ds, precision, &c, false, true) : GOO_OK;
                        }));
  d.gram_key[pi] = key;
  return GOO_OK;
}

// Terms 2k, 2k + 1 of a gradient map: the coefficient parameters of amplitude k.
template <int N>
static void map_coefficients(const DalitzModel& d, GradMap<N>& map) {
  for (int k = d.K - 1; k >= 0; --k) {
    map.add(2 * k + 1, d.par_im[k]);
    map.add(2 * k, d.par_re[k]);
  }
}

template <typename T>
static void fill_args(const DalitzModel& d, const double* theta, int n_params, int64_t n_total, CohArgs<T>& a) {
  std::memset(&a, 0, sizeof a);
  a.nbw = d.nbw;
  a.K = d.K;
  a.has_nr = d.has_nr ? 1 : 0;
  a.n_params = n_params;
  a.n_total = n_total;
  for (int k = 0; k < d.K; ++k) {
    double re, im;
    coef(d, theta, k, re, im);
    a.cr[k] = (T)re;
    a.ci[k] = (T)im;
  }
  a.map.clear();
  if (d.floating)
    for (int k = d.nbw - 1; k >= 0; --k) {
      a.map.add(2 * (d.K + k) + 1, d.par_w[k]);
      a.map.add(2 * (d.K + k), d.par_m0[k]);
    }
  map_coefficients(d, a.map);
  fill_jacobian(d, theta, a);
}

// The normalisation at theta from the host copy of the Gram matrix (ensure_gram keeps it
// current), in FP64 at the precision-rounded coefficients the kernel uses:
//   v_k = sum_l G_kl conj(c_l),  N = sum_k Re(c_k v_k),  dN / d Re c_k = 2 Re v_k,
//   dN / d Im c_k = -2 Im v_k.
template <typename T>
static void coh_norm_terms(const DalitzModel& d, const double* G, CohArgs<T>& a) {
  const int K = d.K;
  double vr[kMaxAmp], vi[kMaxAmp], N = 0.0;
  for (int k = 0; k < K; ++k) {
    vr[k] = vi[k] = 0.0;
    for (int l = 0; l < K; ++l) {
      const double gr = G[2 * (k * K + l)], gi = G[2 * (k * K + l) + 1];
      const double clr = (double)a.cr[l], cli = (double)a.ci[l];
      vr[k] += gr * clr + gi * cli;
      vi[k] += gi * clr - gr * cli;
    }
    N += (double)a.cr[k] * vr[k] - (double)a.ci[k] * vi[k];
  }
  const double invN = 1.0 / N;
  for (int k = 0; k < K; ++k) {
    a.nrm_vr[k] = 2.0 * vr[k] * invN;
    a.nrm_vi[k] = 2.0 * vi[k] * invN;
  }
  a.nrm_N = N;
  a.nrm_logN = std::log(N);
}

constexpr int kMaxDevicesCoh = 64;

template <int KB, bool GRAD>
static int launch_coh_staged(goo_model* m, const void* cache, const goo_dataset* ds, int64_t begin, int64_t end,
                             const double* theta, int out_mode, int pi) {
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  const int planes = (d.nbw + 1) / 2;
  const size_t smem = (size_t)kCohStages<KB> * planes * kCohTile * sizeof(float4);
  static bool configured[kMaxDevicesCoh] = {};
  if (ctx->device < 0 || ctx->device >= kMaxDevicesCoh) return set_error(GOO_ERR_ARG, "device %d", ctx->device);
  if (!configured[ctx->device]) {
    GOO_CUDA_TRY(cudaFuncSetAttribute(coh_nll_staged_kernel<KB, GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)((size_t)kCohStages<KB> * ((KB + 1) / 2) * kCohTile * sizeof(float4))));
    configured[ctx->device] = true;
  }
  const int occ = cached_occupancy((const void*)coh_nll_staged_kernel<KB, GRAD>, ctx->device, kStagedBlock, smem);
  const int64_t tiles = (end + kCohTile - 1) / kCohTile - begin / kCohTile;
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)ctx->num_sms * occ));
  constexpr int NS = CohLanes<float, KB, GRAD>::NS;
  GOO_TRY(ensure_partials(ctx, (size_t)nb * NS));
  CohArgs<float> a;
  fill_args<float>(d, theta, m->n_params, ds->n, a);
  coh_norm_terms<float>(d, d.gram_host[pi], a);
  {
    LaunchScope ls(ctx, GRAD ? "coh_nll_grad_f32" : "coh_nll_f32");
    GOO_CUDA_TRY(launch_early(coh_nll_staged_kernel<KB, GRAD>, nb, kStagedBlock, smem, ctx->stream, a, (const float4*)cache,
                              begin, end, ctx->scratch.partials, ctx->scratch.counters, ctx->scratch.result_out, out_mode));
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

template <int KB, bool GRAD>
static int launch_coh_f64(goo_model* m, const void* cache, const goo_dataset* ds, int64_t begin, int64_t end,
                          const double* theta, int out_mode, int pi) {
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  const int occ = cached_occupancy((const void*)coh_nll_f64_kernel<KB, GRAD>, ctx->device, kBlock, 0);
  const int nb = grid_blocks(ctx, end - begin, occ);
  constexpr int NS = CohLanes<double, KB, GRAD>::NS;
  GOO_TRY(ensure_partials(ctx, (size_t)nb * NS));
  CohArgs<double> a;
  fill_args<double>(d, theta, m->n_params, ds->n, a);
  coh_norm_terms<double>(d, d.gram_host[pi], a);
  {
    LaunchScope ls(ctx, GRAD ? "coh_nll_grad_f64" : "coh_nll_f64");
    coh_nll_f64_kernel<KB, GRAD><<<nb, kBlock, 0, ctx->stream>>>(a, (const double2*)cache, begin, end,
                                                                 ctx->scratch.partials, ctx->scratch.counters,
                                                                 ctx->scratch.result_out, out_mode);
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

template <typename T, bool GRAD>
static int launch_coh_sel(goo_model* m, const void* cache, const goo_dataset* ds, int64_t begin, int64_t end,
                          const double* theta, int out_mode, int pi) {
  const bool small = m->dalitz->nbw <= 8;
  if constexpr (sizeof(T) == 4)
    return small ? launch_coh_staged<8, GRAD>(m, cache, ds, begin, end, theta, out_mode, pi)
                 : launch_coh_staged<15, GRAD>(m, cache, ds, begin, end, theta, out_mode, pi);
  else
    return small ? launch_coh_f64<8, GRAD>(m, cache, ds, begin, end, theta, out_mode, pi)
                 : launch_coh_f64<15, GRAD>(m, cache, ds, begin, end, theta, out_mode, pi);
}

// Constants of the floating-lineshape kernels at theta (FP64 on the host, rounded to T):
// the coefficients by slot and, per resonance (mass m0, width Gamma0, spin L, daughters A, B),
//   d(q0^2) / d m0 = (m0^4 - (mA + mB)^2 (mA - mB)^2) / (2 m0^3),
//   rho   = F'(z0) / (2 F(z0)) r^2 d(q0^2) / d m0   (F(z) = 1 + z for L = 1, 9 + 3z + z^2 for
//           L = 2: the squared barrier ratio is F(z0) / F(z); rho = 0 for L = 0),
//   kappa = 2 / m0 - (2L + 1) d(q0^2) / d m0 / (2 q0^2) + 2 rho.
template <typename T>
static void fill_ls(const DalitzModel& d, const double* theta, LsConst<T>& c) {
  std::memset(&c, 0, sizeof c);
  for (int k = 0; k < d.nbw; ++k) {
    double re, im;
    coef(d, theta, k, re, im);
    c.cr[k] = (T)re;
    c.ci[k] = (T)im;
    c.nci[k] = -c.ci[k];
    double mA, mB, mC;
    pair_masses(d, d.pair[k], mA, mB, mC);
    const int L = d.spin[k];
    const double m0 = theta[d.par_m0[k]], g0 = theta[d.par_w[k]];
    const double u = m0 * m0, thrP = (mA + mB) * (mA + mB), thrM = (mA - mB) * (mA - mB);
    const double q0sq = kallen(u, mA * mA, mB * mB) / (4 * u);
    const double dq0sq = (u * u - thrP * thrM) / (2 * m0 * m0 * m0);
    const double r2 = d.r_res * d.r_res, z0 = r2 * q0sq;
    double rho = 0.0;
    if (L == 1) rho = 0.5 / (1.0 + z0) * r2 * dq0sq;
    if (L == 2) rho = 0.5 * (3.0 + 2.0 * z0) / (9.0 + 3.0 * z0 + z0 * z0) * r2 * dq0sq;
    const double kappa = 2.0 / m0 - (2 * L + 1) * dq0sq / (2.0 * q0sq) + 2.0 * rho;
    c.rho[k] = rho;
    c.kappa[k] = kappa;
    c.two_m0[k] = 2.0 * m0;
    c.inv_g0[k] = 1.0 / g0;
  }
}

template <typename T, int KB, bool GRAD>
static int launch_ls(goo_model* m, const goo_dataset* ds, int64_t begin, int64_t end, const double* theta,
                     int out_mode) {
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  constexpr size_t smem = ls_smem<T, KB, GRAD>();
  constexpr int NS = LsLanes<KB, GRAD>::NS;
  constexpr int NT = kLsBlockOf<KB>;
  const void* fn = (const void*)coh_ls_kernel<T, KB, GRAD>;
  GOO_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  const int64_t cap = (int64_t)ctx->num_sms * cached_occupancy(fn, ctx->device, NT, smem);
  // blocks in proportion to the points, at least one each, no more than there are steps
  constexpr int per = sizeof(T) == 4 ? 2 : 1;
  auto steps = [](int64_t n) { return (n / per + 1 + NT) / NT; };
  const int64_t n_mc = d.mc->n, n_ev = end - begin;
  const int64_t want_mc = std::max<int64_t>(1, (int64_t)((double)cap * n_mc / (double)(n_mc + n_ev) + 0.5));
  const int nb_mc = (int)std::min<int64_t>(std::min<int64_t>(want_mc, cap - 1), steps(n_mc));
  const int nb_ev = (int)std::min<int64_t>(cap - nb_mc, steps(n_ev));
  GOO_TRY(ensure_partials(ctx, (size_t)(nb_mc + nb_ev) * NS));
  CohArgs<T> a;
  fill_args<T>(d, theta, m->n_params, ds->n, a);
  LsConst<T> c;
  fill_ls<T>(d, theta, c);
  if (d.has_nr) {
    double re, im;
    coef(d, theta, d.nbw, re, im);
    c.cr[KB] = (T)re;
    c.ci[KB] = (T)im;
  }
  auto set = [&](const goo_dataset* s, int64_t b, int64_t e) {
    if constexpr (sizeof(T) == 4) return LsSet<T>{s->d32[d.col12], s->d32[d.col13], b, e, s->n};
    else return LsSet<T>{s->d64[d.col12], s->d64[d.col13], b, e, s->n};
  };
  {
    LaunchScope ls(ctx, sizeof(T) == 4 ? (GRAD ? "coh_ls_grad_f32" : "coh_ls_f32") : (GRAD ? "coh_ls_grad_f64" : "coh_ls_f64"));
    const LsTables<T>* t;
    if constexpr (sizeof(T) == 4) t = &d.ls32;
    else t = &d.ls64;
    coh_ls_kernel<T, KB, GRAD><<<nb_mc + nb_ev, NT, smem, ctx->stream>>>(
        a, c, *t, set(d.mc, 0, n_mc), set(ds, begin, end), nb_mc, ctx->scratch.partials, ctx->scratch.counters,
        ctx->scratch.result_out, out_mode);
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

template <typename T, bool GRAD>
static int launch_ls_sel(goo_model* m, const goo_dataset* ds, int64_t begin, int64_t end, const double* theta,
                         int out_mode) {
  return m->dalitz->nbw <= 8 ? launch_ls<T, 8, GRAD>(m, ds, begin, end, theta, out_mode)
                             : launch_ls<T, 15, GRAD>(m, ds, begin, end, theta, out_mode);
}

// The three MC Gram matrices of the time-dependent three-body model (G_aa, G_bb, G_ab) in
// `precision`, rebuilt when the lineshapes or the MC sample change; a host copy for
// goo_normalise.  `ds` as in ensure_gram, both its caches.
static int ensure_td_grams(goo_model* m, int precision, const goo_dataset* ds = nullptr) {
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  const int pi = precision == GOO_F32 ? 0 : 1;
  if (!d.mc) return set_error(GOO_ERR_STATE, "amplitude model has no MC normalisation sample (goo_model_set_norm)");
  if (d.mc->n < 1) return set_error(GOO_ERR_ARG, "the MC normalisation sample is empty");
  const uint64_t key = d.ls_key ^ (uint64_t)(uintptr_t)d.mc ^ (uint64_t)(pi + 11) ^ d.mc->epoch * 0xd6e8feb86659fd93ull;
  if (d.gram3_key[pi] == key) return GOO_OK;
  const void *ca = nullptr, *cb = nullptr;
  GOO_TRY(ensure_cache(m, d.mc, precision, &ca));
  GOO_TRY(ensure_cache(m, d.mc, precision, &cb, true));
  const void *x[3] = {ca, cb, ca}, *y[3] = {ca, cb, cb};
  GOO_TRY(gram_matrices(ctx, precision, true, 3, x, y, d.mc->n, d.nbw, d.K, d.gram3_host[pi],
                        pi == 0 ? "td3_gram_f32" : "td3_gram_f64", [&]() -> int {
                          const void* c = nullptr;
                          if (!ds) return GOO_OK;
                          GOO_TRY(ensure_cache(m, ds, precision, &c, false, true));
                          return ensure_cache(m, ds, precision, &c, true);
                        }));
  d.gram3_key[pi] = key;
  return GOO_OK;
}

template <typename T>
static void fill_td3(const DalitzModel& d, const double* theta, int n_params, int64_t n_total, Td3Args<T>& a,
                     double t_hi) {
  std::memset(&a, 0, sizeof a);
  for (int k = 0; k < d.K; ++k) {
    const int sl = k < d.nbw ? k : kTd3KB;
    double re, im;
    coef(d, theta, k, re, im);
    a.cr[sl] = (T)re;
    a.ci[sl] = (T)im;
  }
  a.map.clear();
  for (int j = 3; j >= 0; --j) a.map.add(2 * kMaxAmp + j, d.par_t[j]);
  map_coefficients(d, a.map);
  fill_time_coef<T>(a.tc, theta[d.par_t[0]], theta[d.par_t[1]], theta[d.par_t[2]], theta[d.par_t[3]], t_hi);
  a.x = a.tc.x;
  a.y = a.tc.y;
  a.G = a.tc.G;
  a.s = a.tc.s;
  const WeidemanTables& w = weideman();
  a.wN = sizeof(T) == 4 ? kWN32 : kWN64;
  for (int j = 0; j < a.wN; ++j) a.wa[j] = (T)(sizeof(T) == 4 ? w.a32[j] : w.a64[j]);
  a.wL = (T)(sizeof(T) == 4 ? w.L32 : w.L64);
  a.nbw = d.nbw;
  a.K = d.K;
  a.n_params = n_params;
  a.n_total = n_total;
  fill_jacobian(d, theta, a);
}

// The normalisation at theta from the host copies of the three Gram matrices G_aa, G_bb, G_ab
// (ensure_td_grams keeps them current), in FP64 at the precision-rounded parameters the kernel
// uses.  With v_a = G_aa conj(c), v_b = G_bb conj(c), u = G_ab conj(c), w = c^T G_ab:
//   <|A|^2> = Re c.v_a, <|B|^2> = Re c.v_b, <A B*> = c.u,
//   N = (<|A|^2> + <|B|^2>)/2 I_ch + (<|A|^2> - <|B|^2>)/2 I_c + Re<AB*> I_sh + Im<AB*> I_s,
//   d<|A|^2> / d Re c_k = 2 Re v_a,k, / d Im c_k = -2 Im v_a,k;
//   d<AB*> / d Re c_k = u_k + w_k, / d Im c_k = i (u_k - w_k);
// and the time integrals' derivatives for x, y and tau.
template <typename T>
static void td3_norm_terms(const DalitzModel& d, const double* G, Td3Args<T>& a) {
  const int K = d.K;
  const double* Gaa = G;
  const double* Gbb = G + 2 * K * K;
  const double* Gab = G + 4 * K * K;
  auto cf = [&](int j, double& r, double& im) {
    const int sl = j < d.nbw ? j : kTd3KB;
    r = (double)a.cr[sl];
    im = (double)a.ci[sl];
  };
  const double x = (double)a.x, y = (double)a.y, tau = 1.0 / (double)a.G;
  const double iy = 1.0 / (1 - y * y), ix = 1.0 / (1 + x * x);
  const double Ich = tau * iy, Ish = y * tau * iy, Ic = tau * ix, Is = x * tau * ix;
  double var[kMaxAmp], vai[kMaxAmp], vbr[kMaxAmp], vbi[kMaxAmp], ur[kMaxAmp], ui[kMaxAmp], wr[kMaxAmp], wi[kMaxAmp];
  double PA = 0, PB = 0, Xr = 0, Xi = 0;
  for (int k = 0; k < K; ++k) {
    var[k] = vai[k] = vbr[k] = vbi[k] = ur[k] = ui[k] = wr[k] = wi[k] = 0.0;
    for (int l = 0; l < K; ++l) {
      double clr, cli;
      cf(l, clr, cli);
      const double ar_ = Gaa[2 * (k * K + l)], ai_ = Gaa[2 * (k * K + l) + 1];
      const double br_ = Gbb[2 * (k * K + l)], bi_ = Gbb[2 * (k * K + l) + 1];
      const double xr_ = Gab[2 * (k * K + l)], xi_ = Gab[2 * (k * K + l) + 1];
      const double yr_ = Gab[2 * (l * K + k)], yi_ = Gab[2 * (l * K + k) + 1];
      var[k] += ar_ * clr + ai_ * cli;  // G_aa[k][l] conj(c_l)
      vai[k] += ai_ * clr - ar_ * cli;
      vbr[k] += br_ * clr + bi_ * cli;
      vbi[k] += bi_ * clr - br_ * cli;
      ur[k] += xr_ * clr + xi_ * cli;  // G_ab[k][l] conj(c_l)
      ui[k] += xi_ * clr - xr_ * cli;
      wr[k] += clr * yr_ - cli * yi_;  // c_l G_ab[l][k]
      wi[k] += clr * yi_ + cli * yr_;
    }
    double ckr, cki;
    cf(k, ckr, cki);
    PA += ckr * var[k] - cki * vai[k];  // Re(c_k v_a,k)
    PB += ckr * vbr[k] - cki * vbi[k];
    Xr += ckr * ur[k] - cki * ui[k];  // c_k u_k (summed: <A B*>)
    Xi += ckr * ui[k] + cki * ur[k];
  }
  const double N = 0.5 * (PA + PB) * Ich + 0.5 * (PA - PB) * Ic + Xr * Ish + Xi * Is;
  const double invN = 1.0 / N;
  for (int k = 0; k < K; ++k) {
    const double dre = 0.5 * (2 * var[k] + 2 * vbr[k]) * Ich + 0.5 * (2 * var[k] - 2 * vbr[k]) * Ic +
                       (ur[k] + wr[k]) * Ish + (ui[k] + wi[k]) * Is;
    const double dim = 0.5 * (-2 * vai[k] - 2 * vbi[k]) * Ich + 0.5 * (-2 * vai[k] + 2 * vbi[k]) * Ic -
                       (ui[k] - wi[k]) * Ish + (ur[k] - wr[k]) * Is;
    a.nrm_re[k] = dre * invN;
    a.nrm_im[k] = dim * invN;
  }
  a.nrm_N = N;
  a.nrm_logN = std::log(N);
  const double ix2 = ix * ix, iy2 = iy * iy;
  const double dxc = -2 * x * tau * ix2, dxs = tau * (1 - x * x) * ix2;
  const double dych = 2 * y * tau * iy2, dysh = tau * (1 + y * y) * iy2;
  a.nrm_dt[0] = (0.5 * (PA - PB) * dxc + Xi * dxs) * invN;
  a.nrm_dt[1] = (0.5 * (PA + PB) * dych + Xr * dysh) * invN;
  a.nrm_dt[2] = (0.5 * (PA + PB) * iy + 0.5 * (PA - PB) * ix + Xr * y * iy + Xi * x * ix) * invN;
}

template <typename T, bool GRAD>
static int launch_td3(goo_model* m, const goo_dataset* ds, int64_t begin, int64_t end, const double* theta,
                      const void* ca, const void* cb, int out_mode) {
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  const int pi = sizeof(T) == 4 ? 0 : 1;
  const void* fn;
  if constexpr (sizeof(T) == 4) fn = (const void*)td3_nll_f32_kernel<GRAD>;
  else fn = (const void*)td3_nll_f64_kernel<GRAD>;
  const int nb = grid_blocks(ctx, end - begin, cached_occupancy(fn, ctx->device, kBlock, 0));
  constexpr int NS = Td3Lanes<GRAD>::NS;
  GOO_TRY(ensure_partials(ctx, (size_t)nb * NS));
  const Fp64Tables* tables = nullptr;
  if (sizeof(T) == 8) GOO_TRY(fp64_tables(ctx, &tables));
  Td3Args<T> a;
  fill_td3<T>(d, theta, m->n_params, ds->n, a, m->hi[d.col_t]);
  td3_norm_terms<T>(d, d.gram3_host[pi], a);
  {
    LaunchScope ls(ctx, sizeof(T) == 4 ? (GRAD ? "td3_nll_grad_f32" : "td3_nll_f32")
                                       : (GRAD ? "td3_nll_grad_f64" : "td3_nll_f64"));
    if constexpr (sizeof(T) == 4)
      td3_nll_f32_kernel<GRAD><<<nb, kBlock, 0, ctx->stream>>>(a, (const float4*)ca, (const float4*)cb, ds->d32[d.col_t],
                                                               begin, end, ctx->scratch.partials, ctx->scratch.counters,
                                                               ctx->scratch.result_out, out_mode);
    else
      td3_nll_f64_kernel<GRAD><<<nb, kBlock, 0, ctx->stream>>>(a, (const double2*)ca, (const double2*)cb,
                                                               ds->d64[d.col_t], tables, begin, end,
                                                               ctx->scratch.partials, ctx->scratch.counters,
                                                               ctx->scratch.result_out, out_mode);
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

// N of the time-dependent three-body model at theta from the host copy of the Gram matrices.
static double td3_norm_host(const DalitzModel& d, const double* G, const double* theta, bool f32) {
  const int K = d.K;
  auto cf = [&](int k, double& r, double& i) {
    coef(d, theta, k, r, i);
    if (f32) {
      r = (double)(float)r;
      i = (double)(float)i;
    }
  };
  double PA = 0, PB = 0, Xr = 0, Xi = 0;
  for (int k = 0; k < K; ++k)
    for (int l = 0; l < K; ++l) {
      double ckr, cki, clr, cli;
      cf(k, ckr, cki);
      cf(l, clr, cli);
      const double pr = ckr * clr + cki * cli, pim = cki * clr - ckr * cli;  // c_k conj(c_l)
      const double* Gs[3] = {G, G + 2 * K * K, G + 4 * K * K};
      const double gr[3] = {Gs[0][2 * (k * K + l)], Gs[1][2 * (k * K + l)], Gs[2][2 * (k * K + l)]};
      const double gi[3] = {Gs[0][2 * (k * K + l) + 1], Gs[1][2 * (k * K + l) + 1], Gs[2][2 * (k * K + l) + 1]};
      PA += pr * gr[0] - pim * gi[0];
      PB += pr * gr[1] - pim * gi[1];
      Xr += pr * gr[2] - pim * gi[2];
      Xi += pr * gi[2] + pim * gr[2];
    }
  double x = theta[d.par_t[0]], y = theta[d.par_t[1]], tau = theta[d.par_t[2]];
  if (f32) {
    x = (double)(float)x;
    y = (double)(float)y;
    tau = 1.0 / (double)(float)(1.0 / tau);
  }
  const double Ich = tau / (1 - y * y), Ish = y * tau / (1 - y * y), Ic = tau / (1 + x * x), Is = x * tau / (1 + x * x);
  return 0.5 * (PA + PB) * Ich + 0.5 * (PA - PB) * Ic + Xr * Ish + Xi * Is;
}

int build_dalitz_model(goo_ctx* ctx, const goo_node* nodes, int n_nodes, int n_params, int n_obs, const double* lo,
                       const double* hi, goo_model* m) {
  const goo_node& root = nodes[n_nodes - 1];
  if (root.n_child < 1 || root.n_child > kMaxAmp)
    return set_error(GOO_ERR_UNSUPPORTED, "coherent sum of %d amplitudes (1..%d)", root.n_child, kMaxAmp);
  if (n_obs < 2 || root.obs[0] < 0 || root.obs[1] < 0 || root.obs[0] >= n_obs || root.obs[1] >= n_obs)
    return set_error(GOO_ERR_ARG, "coherent node needs observables s12 and s13");
  DalitzModel* d = new DalitzModel();
  m->dalitz = d;
  m->kind = 1;
  d->col12 = root.obs[0];
  d->col13 = root.obs[1];
  if (root.op == GOO_OP_TD3) {
    d->td = true;
    d->col_t = root.ival[0];
    if (n_obs < 3 || d->col_t < 0 || d->col_t >= n_obs || d->col_t == d->col12 || d->col_t == d->col13)
      return set_error(GOO_ERR_ARG, "GOO_OP_TD3 needs a decay-time observable (ival[0]) besides s12 and s13");
    for (int j = 0; j < 4; ++j) {
      if (root.par[j] < 0 || root.par[j] >= n_params)
        return set_error(GOO_ERR_ARG, "GOO_OP_TD3: time parameter %d has index %d", j, root.par[j]);
      d->par_t[j] = root.par[j];
    }
  }
  d->M = root.dval[0];
  d->m1 = root.dval[1];
  d->m2 = root.dval[2];
  d->m3 = root.dval[3];
  d->r_res = root.dval[4];
  d->r_par = root.dval[5];
  if (!(d->M > d->m1 + d->m2 + d->m3) || d->m1 < 0 || d->m2 < 0 || d->m3 < 0)
    return set_error(GOO_ERR_ARG, "parent mass %g below the sum of the daughter masses", d->M);
  auto check_par = [&](int p) { return p >= 0 && p < n_params; };
  // BWs first (in tree order), then the NR amplitude
  for (int pass = 0; pass < 2; ++pass) {
    for (int c = 0; c < root.n_child; ++c) {
      const goo_node& a = nodes[root.child[c]];
      if (a.op != GOO_OP_BW && a.op != GOO_OP_NR)
        return set_error(GOO_ERR_ARG, "coherent child %d has op %d (BW or NR expected)", c, a.op);
      if ((pass == 0) != (a.op == GOO_OP_BW)) continue;
      const int k = d->K++;
      if (!check_par(a.par[2]) || !check_par(a.par[3]))
        return set_error(GOO_ERR_ARG, "amplitude %d has no coefficient parameters", c);
      d->par_re[k] = a.par[2];
      d->par_im[k] = a.par[3];
      if (a.op == GOO_OP_BW) {
        if (!check_par(a.par[0]) || !check_par(a.par[1]))
          return set_error(GOO_ERR_ARG, "BW amplitude %d has no mass/width parameters", c);
        if (a.ival[0] < 0 || a.ival[0] > 2) return set_error(GOO_ERR_UNSUPPORTED, "BW spin %d (0..2)", a.ival[0]);
        if (a.ival[1] < 0 || a.ival[1] > 2) return set_error(GOO_ERR_ARG, "BW pair %d (0..2)", a.ival[1]);
        d->par_m0[k] = a.par[0];
        d->par_w[k] = a.par[1];
        d->spin[k] = a.ival[0];
        d->pair[k] = a.ival[1];
        d->nbw++;
      } else {
        if (d->has_nr) return set_error(GOO_ERR_UNSUPPORTED, "at most one non-resonant amplitude");
        d->has_nr = true;
      }
    }
  }
  if (d->nbw > 15) return set_error(GOO_ERR_UNSUPPORTED, "at most 15 resonances");
  if (d->td && std::fabs(d->m2 - d->m3) > 1e-12 * d->M)
    return set_error(GOO_ERR_ARG, "GOO_OP_TD3: the CP-conjugate particles 2 and 3 need equal masses (%g, %g)", d->m2,
                     d->m3);
  (void)lo;
  (void)hi;
  if (cudaMalloc(&d->dev, sizeof(DalitzDev)) != cudaSuccess) {
    cudaGetLastError();
    return set_error(GOO_ERR_OOM, "cannot allocate the amplitude model");
  }
  m->norm.kind = GOO_NORM_MC;
  (void)ctx;
  return GOO_OK;
}

int dalitz_set_norm(goo_model* m, const goo_norm_spec* spec) {
  if (spec->kind != GOO_NORM_MC || !spec->mc)
    return set_error(GOO_ERR_UNSUPPORTED, "amplitude models are normalised with an MC sample (GOO_NORM_MC)");
  const goo_dataset* mc = spec->mc;
  DalitzModel& d = *m->dalitz;
  if (mc->ctx != m->ctx) return set_error(GOO_ERR_ARG, "MC sample belongs to another context");
  if (mc->ncols <= d.col12 || mc->ncols <= d.col13) return set_error(GOO_ERR_ARG, "MC sample lacks s12/s13 columns");
  d.mc = mc;
  d.gram_key[0] = d.gram_key[1] = 0;
  d.gram3_key[0] = d.gram3_key[1] = 0;
  m->norm = *spec;
  return GOO_OK;
}

void dalitz_free(goo_model* m) {
  DalitzModel* d = m->dalitz;
  if (!d) return;
  if (d->dev) cudaFree(d->dev);
  delete d;
  m->dalitz = nullptr;
}

static double quad_form(const DalitzModel& d, const double* G, const double* theta, bool f32) {
  double N = 0.0;
  for (int k = 0; k < d.K; ++k)
    for (int l = 0; l < d.K; ++l) {
      double ckr, cki, clr, cli;
      coef(d, theta, k, ckr, cki);
      coef(d, theta, l, clr, cli);
      if (f32) {
        ckr = (double)(float)ckr;
        cki = (double)(float)cki;
        clr = (double)(float)clr;
        cli = (double)(float)cli;
      }
      const double gr = G[2 * (k * d.K + l)], gi = G[2 * (k * d.K + l) + 1];
      // Re(c_k conj(c_l) G_kl)
      const double pr = ckr * clr + cki * cli, pim = cki * clr - ckr * cli;
      N += pr * gr - pim * gi;
    }
  return N;
}

int dalitz_normalise(goo_model* m, const double* theta, int precision, double* norm_out) {
  GOO_TRY(dalitz_constants(m, theta));
  if (m->dalitz->td) {
    GOO_TRY(ensure_td_grams(m, precision));
    norm_out[0] = td3_norm_host(*m->dalitz, m->dalitz->gram3_host[precision == GOO_F32 ? 0 : 1], theta,
                                precision == GOO_F32);
    return GOO_OK;
  }
  GOO_TRY(ensure_gram(m, precision));
  const int pi = precision == GOO_F32 ? 0 : 1;
  norm_out[0] = quad_form(*m->dalitz, m->dalitz->gram_host[pi], theta, precision == GOO_F32);
  return GOO_OK;
}

int dalitz_nll(goo_model* m, const goo_dataset* ds, int64_t begin, int64_t end, const double* theta, int precision,
               bool grad, double* out, int out_mode) {
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  // the record goes to the mapped host copy; the host polls its fields
  MappedResult mapped(ctx);
  const int P = m->n_params;
  if (ds->ncols <= d.col12 || ds->ncols <= d.col13) return set_error(GOO_ERR_ARG, "dataset lacks s12/s13 columns");
  GOO_TRY(dalitz_constants(m, theta));
  const int nout = (out_mode == 0 ? 2 : 3) + P;
  if (d.td) {
    // time-dependent three-body model: amplitude caches at the event and the exchanged point
    if (ds->ncols <= d.col_t) return set_error(GOO_ERR_ARG, "dataset lacks the decay-time column");
    GOO_TRY(ensure_td_grams(m, precision, end > begin ? ds : nullptr));
    if (end <= begin) {
      for (int i = 0; i < nout; ++i) out[i] = 0.0;
      return GOO_OK;
    }
    const void *ca = nullptr, *cb = nullptr;
    GOO_TRY(ensure_cache(m, ds, precision, &ca));
    GOO_TRY(ensure_cache(m, ds, precision, &cb, true));
    if (precision == GOO_F32) {
      GOO_TRY((grad ? launch_td3<float, true>(m, ds, begin, end, theta, ca, cb, out_mode)
                    : launch_td3<float, false>(m, ds, begin, end, theta, ca, cb, out_mode)));
    } else {
      GOO_TRY((grad ? launch_td3<double, true>(m, ds, begin, end, theta, ca, cb, out_mode)
                    : launch_td3<double, false>(m, ds, begin, end, theta, ca, cb, out_mode)));
    }
  } else if (d.floating) {
    // no cache and no Gram matrix: MC points and events in one launch, lineshape gradients included
    if (!d.mc) return set_error(GOO_ERR_STATE, "amplitude model has no MC normalisation sample (goo_model_set_norm)");
    if (d.mc->n < 1) return set_error(GOO_ERR_ARG, "the MC normalisation sample is empty");
    if (end <= begin) {
      for (int i = 0; i < nout; ++i) out[i] = 0.0;
      return GOO_OK;
    }
    if (precision == GOO_F32) {
      GOO_TRY((grad ? launch_ls_sel<float, true>(m, ds, begin, end, theta, out_mode)
                    : launch_ls_sel<float, false>(m, ds, begin, end, theta, out_mode)));
    } else {
      GOO_TRY((grad ? launch_ls_sel<double, true>(m, ds, begin, end, theta, out_mode)
                    : launch_ls_sel<double, false>(m, ds, begin, end, theta, out_mode)));
    }
  } else {
  GOO_TRY(ensure_gram(m, precision, end > begin ? ds : nullptr));
  const int pi = precision == GOO_F32 ? 0 : 1;
  if (end <= begin) {
    for (int i = 0; i < nout; ++i) out[i] = 0.0;
    return GOO_OK;
  }
  const void* cache = nullptr;
  GOO_TRY(ensure_cache(m, ds, precision, &cache));
  if (precision == GOO_F32) {
    GOO_TRY((grad ? launch_coh_sel<float, true>(m, cache, ds, begin, end, theta, out_mode, pi)
                  : launch_coh_sel<float, false>(m, cache, ds, begin, end, theta, out_mode, pi)));
  } else {
    GOO_TRY((grad ? launch_coh_sel<double, true>(m, cache, ds, begin, end, theta, out_mode, pi)
                  : launch_coh_sel<double, false>(m, cache, ds, begin, end, theta, out_mode, pi)));
  }
  }
  return read_result_mapped(ctx, nout, out);
}

int dalitz_eval_logf(goo_model* m, const goo_dataset* ds, const double* theta, int precision, double* logf_dev) {
  DalitzModel& d = *m->dalitz;
  goo_ctx* ctx = m->ctx;
  if (d.td) return set_error(GOO_ERR_UNSUPPORTED, "goo_eval_logf of the time-dependent three-body model");
  if (ds->ncols <= d.col12 || ds->ncols <= d.col13) return set_error(GOO_ERR_ARG, "dataset lacks s12/s13 columns");
  GOO_TRY(dalitz_constants(m, theta));
  GOO_TRY(ensure_gram(m, precision));
  if (ds->n == 0) return GOO_OK;
  const int pi = precision == GOO_F32 ? 0 : 1;
  const double logN = std::log(quad_form(d, d.gram_host[pi], theta, precision == GOO_F32));
  const void* cache = nullptr;
  GOO_TRY(ensure_cache(m, ds, precision, &cache));
  const int nb = grid_blocks(ctx, ds->n, 4);
  LaunchScope ls(ctx, "coh_logf");
  if (precision == GOO_F32) {
    CohArgs<float> a;
    fill_args<float>(d, theta, m->n_params, ds->n, a);
    if (d.nbw <= 8) coh_logf_kernel<float, 8><<<nb, kBlock, 0, ctx->stream>>>(a, cache, logN, logf_dev);
    else coh_logf_kernel<float, 15><<<nb, kBlock, 0, ctx->stream>>>(a, cache, logN, logf_dev);
  } else {
    CohArgs<double> a;
    fill_args<double>(d, theta, m->n_params, ds->n, a);
    if (d.nbw <= 8) coh_logf_kernel<double, 8><<<nb, kBlock, 0, ctx->stream>>>(a, cache, logN, logf_dev);
    else coh_logf_kernel<double, 15><<<nb, kBlock, 0, ctx->stream>>>(a, cache, logN, logf_dev);
  }
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

// Host copies of the Gram matrix (K x K complex, model amplitude order: resonances in tree
// order, then the non-resonant amplitude) and of the per-event amplitude cache (test access).
int dalitz_gram(goo_model* m, const double* theta, int precision, double* out, int* K_out) {
  if (m->dalitz->td) return set_error(GOO_ERR_UNSUPPORTED, "goo_gram: the time-dependent three-body model has three");
  GOO_TRY(dalitz_constants(m, theta));
  GOO_TRY(ensure_gram(m, precision));
  const int pi = precision == GOO_F32 ? 0 : 1;
  const int K = m->dalitz->K;
  std::memcpy(out, m->dalitz->gram_host[pi], sizeof(double) * 2 * K * K);
  *K_out = K;
  return GOO_OK;
}

int dalitz_amplitudes(goo_model* m, const goo_dataset* ds, const double* theta, int precision, const void** cache,
                      int* nbw) {
  GOO_TRY(dalitz_constants(m, theta));
  GOO_TRY(ensure_cache(m, ds, precision, cache));
  *nbw = m->dalitz->nbw;
  GOO_CUDA_TRY(cudaStreamSynchronize(m->ctx->stream));
  return GOO_OK;
}

int dalitz_cache(goo_model* m, const goo_dataset* ds, int precision, const void** cache) {
  return ensure_cache(m, ds, precision, cache);
}

int dalitz_server_info(goo_model* m, const double* theta, AmpModelInfo* info) {
  if (m->kind != 1) return set_error(GOO_ERR_STATE, "toy server needs an amplitude model");
  if (m->dalitz->td) return set_error(GOO_ERR_UNSUPPORTED, "toy server of the time-dependent three-body model");
  if (m->dalitz->polar) return set_error(GOO_ERR_UNSUPPORTED, "toy server with polar coefficients");
  GOO_TRY(dalitz_constants(m, theta));
  GOO_TRY(ensure_gram(m, GOO_F32));
  GOO_TRY(dalitz_dev(m));
  const DalitzModel& d = *m->dalitz;
  info->dalitz_dev = d.dev;
  info->gram_host = d.gram_host[0];
  info->K = d.K;
  info->nbw = d.nbw;
  info->has_nr = d.has_nr ? 1 : 0;
  for (int k = 0; k < d.K; ++k) {
    info->par_re[k] = d.par_re[k];
    info->par_im[k] = d.par_im[k];
  }
  info->M = d.M;
  info->m1 = d.m1;
  info->m2 = d.m2;
  info->m3 = d.m3;
  info->lo12 = (d.m1 + d.m2) * (d.m1 + d.m2);
  info->hi12 = (d.M - d.m3) * (d.M - d.m3);
  info->lo13 = (d.m1 + d.m3) * (d.m1 + d.m3);
  info->hi13 = (d.M - d.m2) * (d.M - d.m2);
  return GOO_OK;
}

}  // namespace goo

namespace goo {
int dalitz_set_lineshapes(goo_model* m, int mode) {
  if (mode != GOO_LINESHAPE_CACHED && mode != GOO_LINESHAPE_FLOATING)
    return set_error(GOO_ERR_ARG, "goo_model_set_lineshapes: mode %d", mode);
  if (m->dalitz->td && mode == GOO_LINESHAPE_FLOATING)
    return set_error(GOO_ERR_UNSUPPORTED, "floating lineshapes of the time-dependent three-body model");
  m->dalitz->floating = mode == GOO_LINESHAPE_FLOATING;
  return GOO_OK;
}

bool dalitz_lineshape_param(const goo_model* m, int p) {
  const DalitzModel& d = *m->dalitz;
  for (int k = 0; k < d.nbw; ++k)
    if (d.par_m0[k] == p || d.par_w[k] == p) return true;
  return false;
}

bool dalitz_floating(const goo_model* m) { return m->dalitz->floating; }

int dalitz_set_coefficients(goo_model* m, int form) {
  if (form != GOO_COEF_CARTESIAN && form != GOO_COEF_POLAR)
    return set_error(GOO_ERR_ARG, "goo_model_set_coefficients: form %d", form);
  m->dalitz->polar = form == GOO_COEF_POLAR;
  return GOO_OK;
}
bool dalitz_time_dependent(const goo_model* m) { return m->dalitz->td; }
}  // namespace goo
