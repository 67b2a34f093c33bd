// Instantiates part of the spin-summation kernels (see ss_k2.cuh).
#include "ss_k2.cuh"

namespace ss {

bool launch_k2t_d4(const KParams& kp, int ar, cudaStream_t st, cudaError_t* e);

cudaError_t launch_k2_d4_f32(const KParams& kp, cudaStream_t st) {
  cudaError_t e;
  if (launch_k2t_d4(kp, AR_F32, st, &e)) return e;  // 16-byte strides, no beta term
  return launch_k2_impl<4, AR_F32, float>(kp, st);
}
}  // namespace ss
