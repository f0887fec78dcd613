// gram.cuh -- MC Gram matrices of the amplitude models from the amplitude caches:
// G_kl = mean over the sample of X_k conj(Y_l), X and Y two caches of the same events (the same one
// for a Hermitian matrix, of which only the upper triangle is summed).
//
// The matrix is cut into tiles of 4 rows and 8 columns (FP32: 4 and 4).  A block takes one tile and a share of
// the events and keeps the tile's complex sums in registers, so an event's amplitudes are read once for
// all of the tile's products; one block per SM (the sums fill the register file), the SMs
// divided over the tiles in proportion to their products.  One block per row that re-read the whole
// cache for every row and added with scalar Kahan sums took 128 us for 1M points of 9
// amplitudes, this kernel 35 us (64 MB: 9.4 us; some 14 us are launch, reduction and result); the three 16 x 16 matrices of the time-dependent
// three-body model, one block per element with FP64 sums before, 16 ms, now 0.9 ms.
//
// FP32: every event's product is added with Kahan's compensation, real and imaginary part as one packed pair
// (sums and remainders of a 4 x 4 tile take 64 registers), so the sums' error is that of the products'
// rounding, 1e-10 of the mean magnitude at 1M points.  Sums of 16 events run in plain FMAs before a
// compensated addition in shared memory were 8 us faster per scan of three points (320 against 328) and off by
// 1e-9 to 3e-9.  EXACT (the time-dependent three-body model, whose sums were FP64): every product and its rounding
// error (an FMA gives it) is added with compensation, so the result is that of
// FP64 products and sums to 2^-45.  FP64: FMA chains (bound by the FP64 pipe).
// Each tile's last block adds its blocks' sums in block order; results are bitwise repeatable.
#pragma once

#include <functional>

#include "common.cuh"

namespace goo {

constexpr int kGramRows = 4;
template <typename T, bool EXACT>
constexpr int kGramCols = sizeof(T) == 4 && !EXACT ? 4 : 8;
constexpr int kGramTiles = 24;
template <typename T, bool EXACT>
constexpr int kGramLanes = 2 * kGramRows * kGramCols<T, EXACT>;  // lane 2 (k kGramCols + l) + (0: re, 1: im)
// then the rows' own sums (the constant amplitude's column)
template <typename T, bool EXACT>
constexpr int kGramAll = kGramLanes<T, EXACT> + 2 * kGramRows;
constexpr int kGramTickets = 16;  // the tiles' tickets: counters[kGramTickets ..)
// FP32: events requested ahead; a diagonal tile's third and fourth cost registers that 16 warps do not have
// (333 us per scan)
constexpr int kGramAhead = 2;
// threads per block: the most whose sums fit in registers (FP32 in 384 threads: 333 us per scan)
template <typename T, bool EXACT>
constexpr int kGramBlock = sizeof(T) == 8 ? 256 : EXACT ? 384 : 512;
template <typename T, bool EXACT>
constexpr size_t kGramSmem = (size_t)kGramAll<T, EXACT> * kGramBlock<T, EXACT> * sizeof(ddf);

struct GramArgs {
  const void *x[3], *y[3];  // caches of up to three matrices
  int64_t n;
  int nbw, K, ntiles;       // cached amplitudes; K = nbw + 1 with the constant amplitude 1 last
                            // (Hermitian matrices only: its column is the rows' own sums)
  struct Tile {
    int src, r0, c0, diag;  // matrix, first row and column; diag: Hermitian, elements left of the diagonal skipped
    int blk0, nblk;         // its blocks
  } tile[kGramTiles];
};

template <typename T>
struct GramAmp;
template <>
struct GramAmp<float> {
  using V = float2;
  // amplitudes [first, first + N) of event i (N even, first a multiple of 4); those beyond nbw are 0
  template <int N>
  static __device__ __forceinline__ void load(const void* cache, int64_t n, int64_t i, int first, int nbw,
                                              float2 (&a)[N]) {
#pragma unroll
    for (int q = 0; q < N / 2; ++q) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (first + 2 * q < nbw) v = __ldg((const float4*)cache + (int64_t)(first / 2 + q) * n + i);
      a[2 * q] = make_float2(v.x, v.y);
      a[2 * q + 1] = make_float2(v.z, v.w);
    }
  }
};
template <>
struct GramAmp<double> {
  using V = double2;
  template <int N>
  static __device__ __forceinline__ void load(const void* cache, int64_t n, int64_t i, int first, int nbw,
                                              double2 (&a)[N]) {
#pragma unroll
    for (int q = 0; q < N; ++q) {
      a[q] = make_double2(0.0, 0.0);
      if (first + q < nbw) a[q] = __ldg((const double2*)cache + (int64_t)(first + q) * n + i);
    }
  }
};

// One complex sum in registers: x conj(y), or x itself (y = 1).
template <typename T, bool EXACT>
struct GramSum;
template <>
struct GramSum<float, false> {
  float2 s, c;  // (re, im): the sums, and what their roundings left out
  __device__ __forceinline__ void clear() { s = c = make_float2(0.f, 0.f); }
  __device__ __forceinline__ void step(float2 y) {
    const float2 t = pk::add(s, y);
    c = pk::sub(y, pk::sub(t, s));
    s = t;
  }
  __device__ __forceinline__ void mul_add(float2 x, float2 y) {
    step(pk::fma(pk::splat(x.y), make_float2(y.y, y.x), pk::fma(pk::splat(x.x), make_float2(y.x, -y.y), c)));
  }
  __device__ __forceinline__ void add(float2 x) { step(pk::add(x, c)); }
  __device__ __forceinline__ ddf dre() const { return dd_make(s.x, c.x); }
  __device__ __forceinline__ ddf dim() const { return dd_make(s.y, c.y); }
};
template <>
struct GramSum<float, true> {
  Kahan re_, im_;
  __device__ __forceinline__ void clear() { re_ = im_ = Kahan{}; }
  static __device__ __forceinline__ void product(Kahan& s, float a, float b) {
    const float p = __fmul_rn(a, b);
    s.add(p);
    s.c -= fmaf(a, b, -p);
  }
  __device__ __forceinline__ void mul_add(float2 x, float2 y) {
    product(re_, x.x, y.x);
    product(re_, x.y, y.y);
    product(im_, x.y, y.x);
    product(im_, -x.x, y.y);
  }
  __device__ __forceinline__ void add(float2 x) {
    re_.add(x.x);
    im_.add(x.y);
  }
  __device__ __forceinline__ ddf dre() const { return re_.value(); }
  __device__ __forceinline__ ddf dim() const { return im_.value(); }
};
template <>
struct GramSum<double, false> {
  double re, im;
  __device__ __forceinline__ void clear() { re = im = 0.0; }
  __device__ __forceinline__ void mul_add(double2 x, double2 y) {
    re = ::fma(x.x, y.x, ::fma(x.y, y.y, re));
    im = ::fma(x.y, y.x, ::fma(-x.x, y.y, im));
  }
  __device__ __forceinline__ void add(double2 x) {
    re += x.x;
    im += x.y;
  }
  __device__ __forceinline__ ddf dre() const { return dd_from_double(re); }
  __device__ __forceinline__ ddf dim() const { return dd_from_double(im); }
};

template <typename T, bool EXACT>
struct GramAcc {
  GramSum<T, EXACT> m[kGramRows][kGramCols<T, EXACT>], row[kGramRows];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int k = 0; k < kGramRows; ++k) {
      row[k].clear();
#pragma unroll
      for (int l = 0; l < kGramCols<T, EXACT>; ++l) m[k][l].clear();
    }
  }
};

// The thread's sums over its events into its column of s (kGramAll lanes of kGramBlock<T, EXACT> double-floats).
template <typename T, bool EXACT, bool DIAG>
__device__ __forceinline__ void gram_tile_sums(const GramArgs& A, const GramArgs::Tile& t, int64_t i, int64_t stride,
                                               ddf* s) {
  using V = typename GramAmp<T>::V;
  constexpr int COLS = kGramCols<T, EXACT>;
  const void *xc = A.x[t.src], *yc = A.y[t.src];
  GramAcc<T, EXACT> acc;
  acc.clear();
  auto lane = [&](int j) -> ddf& { return s[j * kGramBlock<T, EXACT>]; };
  // the D events ahead are requested before this one's products; a diagonal tile's rows are its first columns
  constexpr int D = sizeof(T) == 4 && !EXACT ? kGramAhead : 1;
  V nx[D][kGramRows], ny[D][COLS];
  auto fetch = [&](int b, int64_t j) {
    if (j >= A.n) return;
    if (!DIAG) GramAmp<T>::load(xc, A.n, j, t.r0, A.nbw, nx[b]);
    GramAmp<T>::load(yc, A.n, j, t.c0, A.nbw, ny[b]);
  };
  auto event = [&](int b) {
#pragma unroll
    for (int l = 0; l < COLS; ++l) {
      if (t.c0 + l >= A.nbw) break;  // uniform
#pragma unroll
      for (int k = 0; k < kGramRows; ++k)
        if (!DIAG || l >= k) acc.m[k][l].mul_add(DIAG ? ny[b][k] : nx[b][k], ny[b][l]);
    }
    if (DIAG) {
#pragma unroll
      for (int k = 0; k < kGramRows; ++k) acc.row[k].add(ny[b][k]);
    }
  };
  if constexpr (D > 1) {
#pragma unroll
    for (int e = 0; e < D; ++e) fetch(e, i + e * stride);
#pragma unroll 1
    for (; i < A.n; i += D * stride) {
#pragma unroll
      for (int e = 0; e < D; ++e) {
        if (i + e * stride >= A.n) break;
        event(e);
        fetch(e, i + (D + e) * stride);
      }
    }
  } else {
    for (; i < A.n; i += stride) {
      fetch(0, i);
      event(0);
    }
  }
#pragma unroll
  for (int k = 0; k < kGramRows; ++k) {
#pragma unroll
    for (int l = 0; l < COLS; ++l) {
      lane(2 * (k * COLS + l)) = acc.m[k][l].dre();
      lane(2 * (k * COLS + l) + 1) = acc.m[k][l].dim();
    }
    lane(kGramLanes<T, EXACT> + 2 * k) = acc.row[k].dre();
    lane(kGramLanes<T, EXACT> + 2 * k + 1) = acc.row[k].dim();
  }
}

// out_host[src]: the K x K matrices (re, im interleaved), in mapped host memory.
template <typename T, bool EXACT>
__global__ void __launch_bounds__(kGramBlock<T, EXACT>, 1) gram_tile_kernel(const __grid_constant__ GramArgs A, float2* partials,
                                                              unsigned* counters, double* out_host) {
  constexpr int COLS = kGramCols<T, EXACT>, LANES = kGramLanes<T, EXACT>, ALL = kGramAll<T, EXACT>;
  extern __shared__ __align__(16) unsigned char s_gram[];
  __shared__ double s_out[ALL];
  __shared__ ddf s_red[kGramBlock<T, EXACT> / 32];
  int ti = 0;
  while (ti + 1 < A.ntiles && (int)blockIdx.x >= A.tile[ti + 1].blk0) ++ti;
  const GramArgs::Tile t = A.tile[ti];  // in registers
  const int b = blockIdx.x - t.blk0;
  ddf* buf = reinterpret_cast<ddf*>(s_gram);
  const int64_t i0 = b * (int64_t)kGramBlock<T, EXACT> + threadIdx.x, stride = (int64_t)t.nblk * kGramBlock<T, EXACT>;
  grid_dep_wait();  // the caches' kernel
  if (t.diag) gram_tile_sums<T, EXACT, true>(A, t, i0, stride, buf + threadIdx.x);
  else gram_tile_sums<T, EXACT, false>(A, t, i0, stride, buf + threadIdx.x);
  grid_dep_launch();  // what is queued behind may take the SMs that are done
  __syncthreads();
  // lane sums over the threads: one warp per lane at a time, then the warp's tree
  float2* part = partials + (size_t)t.blk0 * ALL;
  const int warp = threadIdx.x / 32, w = threadIdx.x % 32;
  for (int lane = warp; lane < ALL; lane += kGramBlock<T, EXACT> / 32) {
    ddf v = buf[lane * kGramBlock<T, EXACT> + w];
    for (int j = w + 32; j < kGramBlock<T, EXACT>; j += 32) v = dd_add(v, buf[lane * kGramBlock<T, EXACT> + j]);
    v = dd_warp_sum(v);
    if (w == 0) part[(size_t)b * ALL + lane] = make_float2(v.hi, v.lo);
  }
  if (!last_block_ticket(counters + kGramTickets + ti, t.nblk)) return;
  reduce_partials(part, ALL, t.nblk, s_out, s_red, kGramBlock<T, EXACT>);
  if (threadIdx.x == 0) counters[kGramTickets + ti] = 0u;
  const double inv_n = 1.0 / (double)A.n;
  const bool hermitian = A.x[t.src] == A.y[t.src];
  const size_t o = (size_t)t.src * 2 * A.K * A.K;
  auto put = [&](int k, int l, int im, double m) {
    const size_t e = o + 2 * (k * A.K + l) + im;
    *(volatile double*)(out_host + e) = m;
  };
  if (threadIdx.x < LANES) {
    const int p = threadIdx.x / 2, im = threadIdx.x & 1;
    const int k = t.r0 + p / COLS, l = t.c0 + p % COLS;
    if (k < A.nbw && l < A.nbw && !(t.diag && l < k)) {
      const double m = (hermitian && im && k == l) ? 0.0 : s_out[threadIdx.x] * inv_n;
      put(k, l, im, m);
      if (hermitian && k != l) put(l, k, im, im ? -m : m);
    }
  } else if (threadIdx.x < ALL) {
    const int k = t.r0 + (threadIdx.x - LANES) / 2, im = threadIdx.x & 1;
    if (t.diag && A.K > A.nbw && k < A.nbw) {  // the constant amplitude: G_k,nbw = mean X_k
      const double m = s_out[threadIdx.x] * inv_n;
      put(k, A.nbw, im, m);
      put(A.nbw, k, im, im ? -m : m);
    }
    if (t.diag && A.K > A.nbw && t.r0 == 0 && threadIdx.x < LANES + 2) put(A.nbw, A.nbw, im, im ? 0.0 : 1.0);
  }
}

// Sums the nmat (1..3) K x K matrices of the caches x[q], y[q] over n events into `host` (nmat x K x K
// complex): launches the kernel, queues
// what `behind` queues (device work that does not need the matrices, so that it runs while the host
// waits for them and launches what does), and waits for the mapped record.  A matrix of two different caches
// needs both caches' own matrices in the same call.  exact: see above (FP32).
int gram_matrices(goo_ctx* ctx, int precision, bool exact, int nmat, const void* const* x, const void* const* y,
                  int64_t n, int nbw, int K, double* host, const char* name,
                  const std::function<int()>& behind = {});

}  // namespace goo
