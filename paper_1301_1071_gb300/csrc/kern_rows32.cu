// kern_rows32.cu -- launchers of the binary32 row products.
#define TSQR_ROWS32_KERNELS
#include "launch.h"
#include "rows32.cuh"

namespace tsqr {

cudaError_t launch_rowmul_f32_tiles(const float* X, const double* M1, const float* Y, const double* M2, int64_t m,
                                    int n, float* out, cudaStream_t st) {
  const int nin = (X ? 1 : 0) + (Y ? 1 : 0);
  const size_t smem = nin * r32_mat(n) + 2 * r32_tile(n);
  cudaError_t e = allow_smem(k_rowmul_f32, smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0, per = 1;
  const int nt = kR32Ty * r32_tx(n);
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_rowmul_f32, nt, smem)) != cudaSuccess) return e;
  const int64_t tiles = (m + kR32Rows - 1) / kR32Rows, slots = static_cast<int64_t>(sms) * (per < 1 ? 1 : per);
  k_rowmul_f32<<<(unsigned)(tiles < slots ? tiles : slots), nt, smem, st>>>(X, M1, Y, M2, m, n, out);
  return cudaGetLastError();
}

cudaError_t launch_form_q_f32_tiles(float* Y, int64_t m, int n, int64_t b, int B, int64_t bt, int kt, int64_t p,
                                    const double* T, const double* C, int64_t cblocks, cudaStream_t st) {
  const size_t smem = 2 * r32_mat(n) + 2 * r32_tile(n);
  cudaError_t e = allow_smem(k_form_q_f32, smem);
  if (e != cudaSuccess) return e;
  k_form_q_f32<<<(unsigned)p, kR32Ty * r32_tx(n), smem, st>>>(Y, m, n, b, B, (int)bt, kt, T, C, cblocks);
  return cudaGetLastError();
}

}  // namespace tsqr
