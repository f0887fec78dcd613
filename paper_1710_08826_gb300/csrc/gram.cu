// gram.cu -- host side of the MC Gram matrices (gram.cuh): the tiles of a launch, their blocks, and the
// result record.
#include <algorithm>
#include <cstring>

#include "gram.cuh"

namespace goo {

template <typename T, bool EXACT>
static int launch_gram_tiles(goo_ctx* ctx, GramArgs& A, double* out_host, const char* name) {
  const void* fn = (const void*)gram_tile_kernel<T, EXACT>;
  GOO_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGramSmem<T, EXACT>));
  int blocks = 0;
  for (int t = 0; t < A.ntiles; ++t) blocks += A.tile[t].nblk;
  GOO_TRY(ensure_partials(ctx, (size_t)blocks * kGramAll<T, EXACT>));
  LaunchScope ls(ctx, name);
  GOO_CUDA_TRY(launch_early(gram_tile_kernel<T, EXACT>, blocks, kGramBlock<T, EXACT>, kGramSmem<T, EXACT>, ctx->stream, A,
                            ctx->scratch.partials, ctx->scratch.counters, out_host));
  GOO_CUDA_TRY(cudaGetLastError());
  return GOO_OK;
}

int gram_matrices(goo_ctx* ctx, int precision, bool exact, int nmat, const void* const* x, const void* const* y,
                  int64_t n, int nbw, int K, double* host, const char* name,
                  const std::function<int()>& behind) {
  const int fields = nmat * 2 * K * K;
  if (nmat > 3 || fields > kGramRecord) return set_error(GOO_ERR_STATE, "Gram matrices of %d fields", fields);
  Scratch& s = ctx->scratch;
  if (!s.gram_host && cudaHostAlloc(&s.gram_host, kGramRecord * sizeof(double), cudaHostAllocMapped) != cudaSuccess) {
    cudaGetLastError();
    s.gram_host = nullptr;
    return set_error(GOO_ERR_OOM, "cannot allocate the Gram matrix record");
  }
  GramArgs A;
  std::memset(&A, 0, sizeof A);
  A.n = n;
  A.nbw = nbw;
  A.K = K;
  // the record comes back through mapped host memory, polled field by field (read_result_mapped)
  arm_mapped(s.gram_host, fields);
  const int cols = precision == GOO_F32 && !exact ? kGramCols<float, false> : kGramCols<double, false>;
  static_assert(kGramCols<float, true> == kGramCols<double, false>, "two widths of tiles");
  int work[kGramTiles], total = 0;
  for (int q = 0; q < nmat; ++q) {
    A.x[q] = x[q];
    A.y[q] = y[q];
    const bool hermitian = x[q] == y[q];
    for (int r0 = 0; r0 < nbw; r0 += kGramRows)
      for (int c0 = hermitian ? r0 : 0; c0 < nbw; c0 += cols) {
        GramArgs::Tile& t = A.tile[A.ntiles];
        t.src = q;
        t.r0 = r0;
        t.c0 = c0;
        t.diag = hermitian && c0 == r0;
        // its products, and about the cost of six more for reading an event
        work[A.ntiles] = kGramRows * std::min(cols, nbw - c0) - (t.diag ? 6 : 0) + 6;
        total += work[A.ntiles++];
      }
    if (nbw < K && (!hermitian || nbw == 0))  // the constant amplitude's fields, which no tile writes
      for (int k = 0; k < K; ++k)
        for (int c = 0; c < 2; ++c) {
          double* g = s.gram_host + (size_t)q * 2 * K * K;
          g[2 * (k * K + nbw) + c] = g[2 * (nbw * K + k) + c] = (k == nbw && c == 0) ? 1.0 : 0.0;
        }
  }
  if (A.ntiles > 0) {
    const int block = precision == GOO_F64 ? kGramBlock<double, false> : exact ? kGramBlock<float, true> : kGramBlock<float, false>;
    const int64_t most = (n + block - 1) / block;
    int blk = 0;
    for (int t = 0; t < A.ntiles; ++t) {
      A.tile[t].blk0 = blk;
      A.tile[t].nblk = (int)std::max<int64_t>(1, std::min<int64_t>(most, (int64_t)ctx->num_sms * work[t] / total));
      blk += A.tile[t].nblk;
    }
    if (precision == GOO_F64) GOO_TRY((launch_gram_tiles<double, false>(ctx, A, s.gram_host, name)));
    else if (exact) GOO_TRY((launch_gram_tiles<float, true>(ctx, A, s.gram_host, name)));
    else GOO_TRY((launch_gram_tiles<float, false>(ctx, A, s.gram_host, name)));
  }
  const int queued = behind ? behind() : GOO_OK;
  GOO_TRY(read_mapped(ctx, s.gram_host, fields, host));  // in any case: the kernel writes the record
  GOO_TRY(queued);
  // of two different caches: mean X_k conj(1) and mean 1 conj(Y_l) from the caches' own matrices
  for (int q = 0; q < nmat && nbw < K; ++q)
    for (int h = 0; h < nmat; ++h) {
      if (x[q] == y[q] || x[h] != y[h]) continue;
      double *g = host + (size_t)q * 2 * K * K, *m = host + (size_t)h * 2 * K * K;
      for (int k = 0; k < nbw; ++k)
        for (int c = 0; c < 2; ++c) {
          if (x[h] == x[q]) g[2 * (k * K + nbw) + c] = m[2 * (k * K + nbw) + c];
          if (x[h] == y[q]) g[2 * (nbw * K + k) + c] = m[2 * (nbw * K + k) + c];
        }
    }
  return GOO_OK;
}

}  // namespace goo
