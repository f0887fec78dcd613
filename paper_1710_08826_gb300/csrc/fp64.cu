// fp64.cu -- the tables of fp64.cuh, computed on the host in extended precision once per process
// and copied to each context's device on first use.
#include <cmath>

#include "common.cuh"
#include "fp64.cuh"

namespace goo {

static const Fp64Tables& host_tables() {
  static const Fp64Tables t = [] {
    Fp64Tables h;
    for (int j = 0; j < kExpTab; ++j) h.exp2j[j] = (double)std::exp2((long double)j / kExpTab);
    for (int j = 0; j < kLogTab; ++j) {
      h.log_inv[j] = (double)(1.0L / (1.0L + (j + 0.5L) / kLogTab));
      h.log_ref[j] = (double)-std::log((long double)h.log_inv[j]);
    }
    constexpr int N = kErfcxDeg + 1;
    const long double pi = 3.14159265358979323846264338327950288L, half = 0.5L / kErfcxStep;
    for (int i = 0; i < kErfcxTab; ++i) {
      const long double c = (long double)i / kErfcxStep;
      h.node[i] = (double)c;
      // interpolation at the Chebyshev points of [c - 1/64, c + 1/64]: divided differences, then
      // the Newton form expanded in powers of r / half
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
      for (int d = 0; d < N; ++d, scale /= half) h.herfcx[d][i] = (double)(poly[d] * scale);
    }
    return h;
  }();
  return t;
}

int fp64_tables(goo_ctx* ctx, const Fp64Tables** dev) {
  Scratch& s = ctx->scratch;
  if (!s.fp64_tables) {
    void* p = nullptr;
    if (cudaMalloc(&p, sizeof(Fp64Tables)) != cudaSuccess) {
      cudaGetLastError();
      return set_error(GOO_ERR_OOM, "cannot allocate the FP64 function tables");
    }
    const cudaError_t e = cudaMemcpyAsync(p, &host_tables(), sizeof(Fp64Tables), cudaMemcpyHostToDevice, ctx->stream);
    if (e != cudaSuccess) {
      cudaFree(p);
      return set_error(GOO_ERR_CUDA, "FP64 function tables: %s", cudaGetErrorString(e));
    }
    s.fp64_tables = p;
  }
  *dev = (const Fp64Tables*)s.fp64_tables;
  return GOO_OK;
}

}  // namespace goo
