// Instantiates part of the spin-summation kernels (see ss_k2.cuh).
#include "ss_k2.cuh"

namespace ss {

bool launch_k2t_d3(const KParams& kp, int ar, cudaStream_t st, cudaError_t* e);

cudaError_t launch_k2_d3(const KParams& kp, int ar, cudaStream_t st) {
  cudaError_t e;
  if (launch_k2t_d3(kp, ar, st, &e)) return e;  // 16-byte strides, no beta term
  if (ar == AR_EXACT) return launch_k2_impl<3, AR_EXACT, double>(kp, st);
  if (ar == AR_STRICT) return launch_k2_impl<3, AR_STRICT, double>(kp, st);
  return launch_k2_impl<3, AR_F32, float>(kp, st);
}
}  // namespace ss
