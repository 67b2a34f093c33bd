// Instantiates part of the spin-summation kernels (see ss_kernels.cuh): d = 4
// through the transform, with the beta term.
#include "ss_kernels.cuh"

namespace ss {

cudaError_t launch_k1_d4_beta(const KParams& kp, cudaStream_t st) {
  k1_kernel<4, AR_EXACT, 1, double, 1, 1><<<dim3((unsigned)kp.pre[npatterns(4)]), dim3(256), 0, st>>>(kp);
  return cudaGetLastError();
}
}  // namespace ss
