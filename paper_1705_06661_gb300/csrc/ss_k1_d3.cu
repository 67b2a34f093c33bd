// Instantiates part of the spin-summation kernels (see ss_kernels.cuh).
#include "ss_kernels.cuh"

namespace ss {

cudaError_t launch_k1_d3(const KParams& kp, int ar, int vec, cudaStream_t st) {
  if (ar == AR_EXACT) {
    if (vec == 2) launch_k1_bt<3, AR_EXACT, 2, double>(kp, st);
    else launch_k1_bt<3, AR_EXACT, 1, double>(kp, st);
  } else if (ar == AR_STRICT) {
    if (vec == 2) launch_k1_bt<3, AR_STRICT, 2, double>(kp, st);
    else launch_k1_bt<3, AR_STRICT, 1, double>(kp, st);
  } else {
    if (vec == 4) launch_k1_bt<3, AR_F32, 4, float>(kp, st);
    else if (vec == 2) launch_k1_bt<3, AR_F32, 2, float>(kp, st);
    else launch_k1_bt<3, AR_F32, 1, float>(kp, st);
  }
  return cudaGetLastError();
}
}  // namespace ss
