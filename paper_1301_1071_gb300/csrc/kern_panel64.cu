// kern_panel64.cu -- launcher of the panel form of Step 1 (binary64 data).
#define TSQR_PANEL_KERNELS
#include "launch.h"
#include "panel64.cuh"

namespace tsqr {

cudaError_t launch_panel_qr_f64(const PanelCfg& k, const void* A, int64_t m, int n, int64_t b, int kt, int64_t p,
                                void* Y, double* Rst, double* Tst, int32_t* status, cudaStream_t st) {
  if (32 * k.NW > kPdMaxThreads) return cudaErrorInvalidConfiguration;
  cudaError_t e = allow_smem(k_panel_qr_f64, k.smem);
  if (e != cudaSuccess) return e;
  k_panel_qr_f64<<<(unsigned)p, 32 * k.NW, k.smem, st>>>(static_cast<const double*>(A), m, n, (int)b, kt, k.NW, k.NS, k.order, k.sms,
                                                         static_cast<double*>(Y), Rst, Tst, status);
  return cudaGetLastError();
}

}  // namespace tsqr
