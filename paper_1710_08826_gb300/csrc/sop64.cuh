// sop64.cuh -- the FP64 event kernel of the sum-of-products models.
//
// The kernel is bound by the FP64 pipe (fp64.cuh: 16 cycles per warp instruction), so the leaf
// dispatch, column selection, sign tests and table lookups, which run on the other pipes, are free and
// an interpreter is as fast as a kernel specialised for the model; what counts is that no FP64
// slot is spent on an absent leaf, lane or product:
//   - each leaf's case adds its exponent and multiplies its factor r only where it has one, and
//     only the gradient lanes that the leaf has are accumulated;
//   - with two products one exponential, exp(-|a_1 - a_0|), serves both; with one, none is needed;
//   - log S is a running product (LogProduct), 1/S, 1/u and 1/r are third-order reciprocals, exp
//     and log come from shared-memory tables;
//   - a polynomial r that is its product's only one needs no reciprocal: c_k / r is the other factors;
//     an event where a polynomial is exactly 0 is left out of its lanes all the same, like the rest of the product
//     (x times the other factors over S may be any number: where a narrow signal is all that is left, it leaves
//     the float range of the block sums, and to carry the exponent that far costs 10 registers, 448 -> 471 us);
//   - the constant factors of the lanes (1/sigma, 2/m0) are applied once per thread, and the Argus endpoint's
//     derivative is formed from the sums of c_k / u, c_k and c_k u.
// The three-dimensional signal + background model takes 76 slots per event (counted) with the
// gradient; the interpreter it replaces took about 235 (3M events: 1123 us; 481 us with
// nine slots more and two blocks per SM, 436 us with two blocks, now 426 us; 100k events: 50 -> 39 us).
#pragma once

#include "fp64.cuh"
#include "model.cuh"
#include "sop_kernels.cuh"

namespace goo {

// exp(-x) for x >= 0, 0 from 746 on (where exp() gives 0 too: a product that far below another one is all
// there is where the other's weight is 0).  NaN stays NaN: a present
// product whose exponent is NaN or +inf (its integral is negative, or vanishes) makes a difference of exponents
// NaN, and the event then has no density, whatever the other products are.
__device__ __forceinline__ double exp_neg(double x, const ExpTable& tab) {
  const int h = __double2hiint(x);
  if (h >= 0x40875000) return h > 0x7ff00000 ? x : 0.0;
  return exp_tab(-x, tab);
}

// On the integer pipe: x is not zero; the largest exponent of an event's products is a number, not an
// absent product's -1e30 nor infinite.
__device__ __forceinline__ bool nonzero(double x) { return (__double_as_longlong(x) << 1) != 0; }
// a b is not zero; the product itself only where it might leave the normal range
__device__ __forceinline__ bool nonzero_product(double a, double b) {
  const int ea = (__double2hiint(a) >> 20) & 0x7ff, eb = (__double2hiint(b) >> 20) & 0x7ff;
  return (ea != 0 && eb != 0 && ea + eb > 1024) || nonzero(a * b);
}
__device__ __forceinline__ bool usable_exponent(double M) {
  const int h = __double2hiint(M);
  return h < 0 ? (h & 0x7fffffff) < 0x45f00000 : h < 0x7ff00000;
}

// Per leaf slot, kept for the gradient: Gauss (z, z^2), Expo (x, -), Poly2 (x, r), Argus (u, log u).
template <int K, int L, bool GRAD>
__global__ void __launch_bounds__(kBlock, 1)
    sop_event64_kernel(const ModelDev* __restrict__ md, const __grid_constant__ EvConst<double, K, L> P,
                       Cols<double> cols, const Fp64Tables* __restrict__ tables, int64_t begin, int64_t end,
                       float2* partials, unsigned* counters, double* result, int out_mode,
                       const double* __restrict__ wcol) {
  constexpr int NS = EventLanes<double, K, L, GRAD>::NS;
  __shared__ ddf s_red[(kBlock / 32) * NS > kBlock ? (kBlock / 32) * NS : kBlock];
  __shared__ unsigned s_bad[kBlock / 32];
  __shared__ SopTables s_tab;
  load_fp64_tables(s_tab, tables);
  const int nK = P.nK, nobs = P.nobs;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t i = begin + blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  // the next event's columns are requested before this one is evaluated
  double nx[kMaxObs] = {0.0, 0.0, 0.0, 0.0}, nw = 1.0;
  auto fetch = [&](int64_t j) {
    if (j >= end) return;
    nx[0] = cols.c[0][j];
    if (nobs > 1) nx[1] = cols.c[1][j];
    if (nobs > 2) nx[2] = cols.c[2][j];
    if (nobs > 3) nx[3] = cols.c[3][j];
    if (wcol) nw = wcol[j];
  };
  fetch(i);
  // the tables and columns depend on no earlier kernel; the offsets -log N_k do
  grid_dep_wait();
  unsigned one_poly = 0;  // bit k: product k has exactly one polynomial
#pragma unroll
  for (int k = 0; k < K; ++k) {
    int np = 0;
#pragma unroll
    for (int l = 0; l < L; ++l) np += P.leaf[k][l].op == GOO_OP_POLY2;
    one_poly |= (k < nK && np == 1 ? 1u : 0u) << k;
  }
  double off[K], unused_lo[K];
  load_offsets<double, K>(md, off, unused_lo);
  double acc = 0.0, C[K], A[K][L][3];
  LogProduct lp;
  unsigned bad = 0;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    C[k] = 0.0;
#pragma unroll
    for (int l = 0; l < L; ++l) A[k][l][0] = A[k][l][1] = A[k][l][2] = 0.0;
  }
  __syncthreads();
  for (; i < end; i += stride) {
    const double x0 = nx[0], x1 = nx[1], x2 = nx[2], x3 = nx[3], wi = nw;
    fetch(i + stride);
    if (wcol && wi == 0.0) continue;  // an empty bin
    // t: the product's factor without its polynomial where it has just one (q; else 1)
    double a[K], t[K], q[K], d0[K][L], d1[K][L];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      a[k] = -1e30;  // an absent product
      t[k] = 0.0;
      q[k] = 1.0;
      if (k >= nK) continue;
      double ak = off[k], r = 1.0, rq = 1.0;
      bool present = true, has_r = false;
#pragma unroll
      for (int l = 0; l < L; ++l) {
        const LeafReg<double>& F = P.leaf[k][l];
        const double x = pick<double>(F.col, x0, x1, x2, x3);
        d0[k][l] = d1[k][l] = 0.0;
        switch (F.op) {
          case GOO_OP_GAUSS: {
            const double z = (x - F.c[0]) * F.c[1], zz = z * z;
            ak = fma(-0.5, zz, ak);
            d0[k][l] = z;
            d1[k][l] = zz;
            break;
          }
          case GOO_OP_EXPO:
            ak = fma(F.c[0], x, ak);
            d0[k][l] = x;
            break;
          case GOO_OP_POLY2: {
            const double rp = fma(x, fma(F.c[1], x, F.c[0]), 1.0);
            if (one_poly >> k & 1) {
              rq = rp;
            } else {
              r = has_r ? r * rp : rp;
              has_r = true;
              d1[k][l] = rp;
            }
            d0[k][l] = x;
            break;
          }
          case GOO_OP_ARGUS: {
            const double u = (F.c[0] - x) * (F.c[0] + x) * F.c[1];
            r = has_r ? r * x : x;
            has_r = true;
            if (__double_as_longlong(u) > 0) {
              const double lu = log_tab(u, s_tab.log);
              ak = fma(F.c[3], lu, fma(F.c[2], u, ak));
              d0[k][l] = u;
              d1[k][l] = lu;
            } else {
              present = false;
            }
            break;
          }
          default:
            break;
        }
      }
      // r == 0: the product vanishes, whatever its exponent
      if (one_poly >> k & 1) present = present && nonzero_product(r, rq);
      else if (has_r) present = present && nonzero(r);
      a[k] = present ? ak : -1e30;
      t[k] = present ? r : 0.0;
      q[k] = present ? rq : 1.0;
    }
    double M = a[0];
    if (K == 2) {
      if (nK == 2) {
        const double d = a[1] - a[0];
        const int hd = __double2hiint(d);
        const double e = exp_neg(__hiloint2double(hd & 0x7fffffff, __double2loint(d)), s_tab.exp);
        const double te = (hd < 0 ? t[1] : t[0]) * e;
        t[0] = hd < 0 ? t[0] : te;
        t[1] = hd < 0 ? te : t[1];
        M = hd < 0 ? a[0] : a[1];
      }
    } else if (nK > 1) {
#pragma unroll
      for (int k = 1; k < K; ++k) M = a[k] > M ? a[k] : M;
#pragma unroll
      for (int k = 0; k < K; ++k)
        if (k < nK) t[k] *= exp_neg(M - a[k], s_tab.exp);
    }
    double tr[K];  // t without the polynomial
#pragma unroll
    for (int k = 0; k < K; ++k) {
      tr[k] = t[k];
      if (one_poly >> k & 1) t[k] *= q[k];
    }
    double S = P.w_hi[0] * t[0];
#pragma unroll
    for (int k = 1; k < K; ++k)
      if (k < nK) S = fma(P.w_hi[k], t[k], S);
    double invS;
    if (positive_normal(S) && usable_exponent(M)) {
      if (wcol) {
        acc = fma(wi, M + log_tab(S, s_tab.log), acc);
      } else {
        acc += M;
        lp.mul(S);
      }
      invS = rcp64(S);
    } else if (S > 0.0 && M > -1e29 && M < HUGE_VAL) {  // S subnormal or infinite
      acc += wi * (M + log(S));
      invS = 1.0 / S;
    } else {
      ++bad;
      continue;
    }
    if constexpr (GRAD) {
      if (wcol) invS *= wi;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (k >= nK) continue;
        const double ck = t[k] * invS;
        C[k] += ck;
#pragma unroll
        for (int l = 0; l < L; ++l) {
          const LeafReg<double>& F = P.leaf[k][l];
          const double p = d0[k][l], q = d1[k][l];
          switch (F.op) {
            case GOO_OP_GAUSS:  // z, z^2 (times 1 / sigma at the end)
              A[k][l][0] = fma(ck, p, A[k][l][0]);
              A[k][l][1] = fma(ck, q, A[k][l][1]);
              break;
            case GOO_OP_EXPO:
              A[k][l][0] = fma(ck, p, A[k][l][0]);
              break;
            case GOO_OP_POLY2: {  // x / r, x^2 / r
              // t / r is the product's other factors; with several polynomials r = 0 only where the product
              // vanishes (ck = 0) and its reciprocal is not used there
              const double cq = one_poly >> k & 1 ? tr[k] * invS : ck * (nonzero(ck) ? recip(q) : 0.0), cx = cq * p;
              A[k][l][0] += cx;
              A[k][l][1] = fma(cx, p, A[k][l][1]);
              break;
            }
            case GOO_OP_ARGUS:  // 1 / u, u, log u
              A[k][l][0] = fma(ck, nonzero(ck) ? recip(p) : 0.0, A[k][l][0]);
              A[k][l][1] = fma(ck, p, A[k][l][1]);
              A[k][l][2] = fma(ck, q, A[k][l][2]);
              break;
            default:
              break;
          }
        }
      }
    }
  }
  if (!wcol) acc += lp.log_value();
  ddf v[NS];
  v[0] = dd_from_double(acc);
  if constexpr (GRAD) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      v[1 + k] = dd_from_double(C[k]);
#pragma unroll
      for (int l = 0; l < L; ++l) {
        const LeafReg<double>& F = P.leaf[k][l];
        const double s0 = F.op == GOO_OP_GAUSS ? F.c[1] : F.op == GOO_OP_ARGUS ? F.c[4] : 1.0;
        // Argus, d / d m0: sum c_k (1 - u) (p / u + c) from the sums of c_k / u, c_k and c_k u
        if (F.op == GOO_OP_ARGUS)
          A[k][l][0] = fma(F.c[3], A[k][l][0], fma(F.c[2] - F.c[3], C[k], -F.c[2] * A[k][l][1]));
        const double s1 = F.op == GOO_OP_GAUSS ? F.c[1] : 1.0;
        v[1 + K + (k * L + l) * 3] = dd_from_double(A[k][l][0] * s0);
        v[1 + K + (k * L + l) * 3 + 1] = dd_from_double(A[k][l][1] * s1);
        v[1 + K + (k * L + l) * 3 + 2] = dd_from_double(A[k][l][2]);
      }
    }
  }
  event_finish<K, L, GRAD, 0>(v, bad, MdFin{md, nK}, nK, partials, counters, result, out_mode, s_red, s_bad);
}

}  // namespace goo
