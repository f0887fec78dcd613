// fp64.cu -- the tables of fp64.cuh, computed on the host in extended precision once per process
// and copied to each context's device on first use.
#include <cmath>

#include "common.cuh"
#include "fp64.cuh"

namespace goo {

// Coefficients c_d of erfcx(u) / 2 = sum_d c_d r^d, r = u - i / 32, |r| <= 1 / 64, of degree DEG:
// interpolation at the Chebyshev points of the interval, divided differences, then the Newton
// form expanded in powers of r.
template <int DEG>
static void herfcx_coeffs(int i, long double (&out)[DEG + 1]) {
  constexpr int N = DEG + 1;
  const long double pi = 3.14159265358979323846264338327950288L, half = 0.5L / kErfcxStep;
  const long double c = (long double)i / kErfcxStep;
  long double r[N], f[N], poly[N] = {0};
  for (int k = 0; k < N; ++k) {
    r[k] = std::cos(pi * (2 * k + 1) / (2 * N));
    const long double u = c + half * r[k];
    f[k] = 0.5L * std::exp(u * u) * std::erfc(u);
  }
  for (int d = 1; d < N; ++d)
    for (int k = N - 1; k >= d; --k) f[k] = (f[k] - f[k - 1]) / (r[k] - r[k - d]);
  for (int k = N - 1; k >= 0; --k) {  // poly = poly (r - r_k) + f_k
    for (int d = N - 1; d > 0; --d) poly[d] = poly[d - 1] - r[k] * poly[d];
    poly[0] = f[k] - r[k] * poly[0];
  }
  long double scale = 1.0L;
  for (int d = 0; d < N; ++d, scale /= half) out[d] = poly[d] * scale;
}

static const Fp64Tables& host_tables() {
  static const Fp64Tables t = [] {
    Fp64Tables h;
    for (int j = 0; j < kExpTab; ++j) h.exp.exp2j[j] = (double)std::exp2((long double)j / kExpTab);
    for (int j = 0; j < kLogTab; ++j) {
      h.log.inv[j] = (double)(1.0L / (1.0L + (j + 0.5L) / kLogTab));
      h.log.ref[j] = (double)-std::log((long double)h.log.inv[j]);
    }
    for (int i = 0; i < kErfcxTab; ++i) {
      h.erfcx.node[i] = (double)i / kErfcxStep;
      long double c[kErfcxDeg + 1];
      herfcx_coeffs<kErfcxDeg>(i, c);
      for (int d = 0; d <= kErfcxDeg; ++d) h.erfcx.herfcx[d][i] = (double)c[d];
    }
    return h;
  }();
  return t;
}

static const Fp32Tables& host_tables32() {
  static const Fp32Tables t = [] {
    Fp32Tables h;
    for (int i = 0; i < kErfcxTab; ++i) {
      long double c[kErfcxDeg32 + 1];
      herfcx_coeffs<kErfcxDeg32>(i, c);
      for (int d = 0; d <= kErfcxDeg32; ++d) h.herfcx[d][i] = (float)c[d];
    }
    return h;
  }();
  return t;
}

// The device copy *slot of a host table, made on first use.
static int device_tables(goo_ctx* ctx, void** slot, const void* host, size_t bytes) {
  if (*slot) return GOO_OK;
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return set_error(GOO_ERR_OOM, "cannot allocate the function tables");
  }
  const cudaError_t e = cudaMemcpyAsync(p, host, bytes, cudaMemcpyHostToDevice, ctx->stream);
  if (e != cudaSuccess) {
    cudaFree(p);
    return set_error(GOO_ERR_CUDA, "function tables: %s", cudaGetErrorString(e));
  }
  *slot = p;
  return GOO_OK;
}

int fp64_tables(goo_ctx* ctx, const Fp64Tables** dev) {
  GOO_TRY(device_tables(ctx, &ctx->scratch.fp64_tables, &host_tables(), sizeof(Fp64Tables)));
  *dev = (const Fp64Tables*)ctx->scratch.fp64_tables;
  return GOO_OK;
}

int fp32_tables(goo_ctx* ctx, const Fp32Tables** dev) {
  GOO_TRY(device_tables(ctx, &ctx->scratch.fp32_tables, &host_tables32(), sizeof(Fp32Tables)));
  *dev = (const Fp32Tables*)ctx->scratch.fp32_tables;
  return GOO_OK;
}

}  // namespace goo
