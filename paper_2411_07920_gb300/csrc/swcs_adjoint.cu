// Adjoint of the truncated gate sequence ("analytic gradients", Sec. II.B).
//
// With every truncation held as the fixed projector P_g onto its kept set S_g,
//   psi_{g+1} = P_{g+1} U_g psi_g,  U_g = exp(theta_g A_g),  A_g = tau_g - tau_g^dag,
//   nu_M      = P_M (H - E) psi_M,
//   dE/dtheta_g = 2 <nu_{g+1} | A_g U_g psi_g> / <psi_M|psi_M>,
//   nu_g      = P_g U_g^dag nu_{g+1}.
// A gate couples each determinant only with its partner, so on a block {L, U}
// with tau L = s U everything is two amplitudes and two entries of nu: the forward
// pass records the blocks (swcs_gates.cu), the backward pass there rotates nu
// in place.  This file holds what is left around it.
#include <cstdint>
#include <cuda_runtime.h>

#include "swcs_device.cuh"
#include "swcs_kernels.h"

namespace swcs {

namespace {

__global__ void build_index_kernel(const uint64_t* keys, const long long* n_ptr, IdxSlot* tab, uint64_t mask) {
  const long long n = *n_ptr;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    idx_insert(tab, mask, keys[i], (uint64_t)i);
}

__global__ void scale_dtheta_kernel(double* d, int n, const double* acc) {
  const double f = 2.0 / acc[1];
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) d[i] *= f;
}

}  // namespace

cudaError_t launch_build_index(const uint64_t* keys, const long long* n, IdxSlot* tab, uint64_t mask, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(tab, 0xff, (mask + 1) * sizeof(IdxSlot), st);
  if (e != cudaSuccess) return e;
  build_index_kernel<<<608, 256, 0, st>>>(keys, n, tab, mask);
  return cudaGetLastError();
}

cudaError_t launch_scale_dtheta(double* d, int n, const double* acc, cudaStream_t st) {
  scale_dtheta_kernel<<<(n + 255) / 256, 256, 0, st>>>(d, n, acc);
  return cudaGetLastError();
}

}  // namespace swcs
