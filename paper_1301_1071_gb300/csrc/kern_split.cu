// kern_split.cu -- launchers of the binary64 digit-product kernels.
#include "launch.h"
#include "split_kernels.cuh"

namespace tsqr {

cudaError_t launch_rowmul_split(const double* X, const double* M, const double* colsrc, const int* colexp, int64_t m,
                                int n, bool add, double* out, int32_t* status, cudaStream_t st) {
  if (n < 1 || n > kRsMaxN) return cudaErrorInvalidValue;
  const size_t smem = RowSplitSmem(n).total;
  const int KC = split_kc(n);
  auto fn = KC == 1   ? k_rowmul_split<1>
            : KC == 2 ? k_rowmul_split<2>
            : KC == 3 ? k_rowmul_split<3>
                      : k_rowmul_split<4>;
  cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  const int64_t need = (m + kRsRows * (kRsThreads / 32) - 1) / (kRsRows * (kRsThreads / 32));
  const int64_t slots = static_cast<int64_t>(sms) * (KC <= 2 ? 2 : 1);
  fn<<<static_cast<unsigned>(need < slots ? need : slots), kRsThreads, smem, st>>>(X, M, colsrc, colexp, m, n, add,
                                                                                  out, status);
  return cudaGetLastError();
}

cudaError_t launch_form_q_split(double* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt, int64_t p,
                                const double* T, const double* C, int64_t cblocks, bool comp, int32_t* status,
                                cudaStream_t st) {
  if (n < 1 || n > kRsMaxN) return cudaErrorInvalidValue;
  const size_t smem = FormQSplitSmem(n).total;
  const int KC = split_kc(n);
  auto fn = KC == 1   ? k_form_q_split<1>
            : KC == 2 ? k_form_q_split<2>
            : KC == 3 ? k_form_q_split<3>
                      : k_form_q_split<4>;
  cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  fn<<<static_cast<unsigned>(p), kRsThreads, smem, st>>>(Y, m, n, static_cast<int>(b), B, static_cast<int>(bt), kt, T,
                                                         C, cblocks, comp, status);
  return cudaGetLastError();
}

// Tiles per warp: ncg warps share the output tiles of ncg (and ncg / 2)
// column groups; 64-row chunks for n <= 64, 32-row chunks above (the digit
// planes of both operands then fit an SM).
template <class S, bool SYM, bool TM>
static cudaError_t gram_split(const S* X, const S* Y, int64_t m, int n, double* part, int* colexp, int64_t b,
                              int B, int bt, int kt, int64_t p, int64_t work, int64_t* grid_max, cudaStream_t st) {
  const int ncg = (n + 7) / 8;
  const int CR = n <= 64 ? 64 : 32;
  auto fn = n <= 32   ? k_gram_split<S, SYM, TM, 64, 2, 128, SYM ? 3 : 2>
            : n <= 64 ? k_gram_split<S, SYM, TM, 64, SYM ? 3 : 4, 256, 1>
                      : k_gram_split<S, SYM, TM, 32, SYM ? 4 : 7, 416, 1>;
  const size_t smem = GramSplitSmem(n, CR, SYM).total;
  cudaError_t e = allow_smem(fn, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per = 1;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, 32 * ncg, smem)) != cudaSuccess) return e;
  int64_t grid = static_cast<int64_t>(sms) * (per < 1 ? 1 : per);
  grid = grid < work ? grid : work;
  grid = grid < *grid_max ? grid : *grid_max;
  *grid_max = grid;
  fn<<<static_cast<unsigned>(grid), 32 * ncg, smem, st>>>(X, Y, m, n, part, colexp, b, B, bt, kt, p);
  return cudaGetLastError();
}

cudaError_t launch_gram_split(const double* X, const double* Y, int64_t m, int n, int max_parts, int* parts,
                              double* part, int* colexp, cudaStream_t st) {
  if (n < 1 || n > TSQR_NMAX) return cudaErrorInvalidValue;
  const int CR = n <= 64 ? 64 : 32;
  const int64_t chunks = (m + CR - 1) / CR;
  int64_t grid = max_parts;
  const cudaError_t e = X == Y ? gram_split<double, true, false>(X, X, m, n, part, colexp, 0, 0, 0, 1, 0, chunks, &grid, st)
                               : gram_split<double, false, false>(X, Y, m, n, part, colexp, 0, 0, 0, 1, 0, chunks, &grid, st);
  *parts = static_cast<int>(grid);
  return e;
}

cudaError_t launch_gram_split_f32(const float* X, int64_t m, int n, int max_parts, int* parts, double* part,
                                  cudaStream_t st) {
  if (n < 1 || n > TSQR_NMAX) return cudaErrorInvalidValue;
  const int CR = n <= 64 ? 64 : 32;
  int64_t grid = max_parts;
  const cudaError_t e =
      gram_split<float, true, false>(X, X, m, n, part, nullptr, 0, 0, 0, 1, 0, (m + CR - 1) / CR, &grid, st);
  *parts = static_cast<int>(grid);
  return e;
}

cudaError_t launch_gram_t_split(const double* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt, int64_t p,
                                double* T, cudaStream_t st) {
  if (n < 1 || n > TSQR_NMAX) return cudaErrorInvalidValue;
  int64_t grid = 1 << 30;
  return gram_split<double, true, true>(Y, Y, m, n, T, nullptr, b, B, static_cast<int>(bt), kt, p, p * kt, &grid, st);
}

}  // namespace tsqr
