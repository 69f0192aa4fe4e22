// The kernels' Householder scalars (qr_kernels.cuh) on arrays, for a test against
// extended precision: out[4 i ..] = beta, scal, ib, tau of (s2[i], alpha[i]).
#include "qr_kernels.cuh"

__global__ void k_scalars(const double* s2, const double* alpha, int k, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= k) return;
  const tsqr::Reflector<double> f = tsqr::make_reflector64(s2[i], alpha[i]);
  out[4 * i] = f.beta;
  out[4 * i + 1] = f.scal;
  out[4 * i + 2] = f.ib;
  out[4 * i + 3] = f.tau;
}

extern "C" int reflector_scalars(const double* s2, const double* alpha, int k, double* out) {
  k_scalars<<<(k + 127) / 128, 128>>>(s2, alpha, k, out);
  return static_cast<int>(cudaDeviceSynchronize());
}
