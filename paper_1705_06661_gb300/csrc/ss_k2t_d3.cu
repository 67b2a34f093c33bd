// Instantiates the TMA-fed tiled kernel for d = 3 (see ss_k2t.cuh).
#include "ss_k2t.cuh"

namespace ss {

// FP64: 24 KB stages, four per CTA and two CTAs per SM (A[544]^3: 426 us at that time, 406 now; three by three
// 448, two groups of eight warps on four stages 445, on nine stages of one CTA 641)
bool launch_k2t_d3(const KParams& kp, int ar, cudaStream_t st, cudaError_t* e) {
  if (ar == AR_EXACT) return launch_k2t<3, AR_EXACT, 4, 2, double>(kp, st, e);
  if (ar == AR_F32) return launch_k2t<3, AR_F32, 4, 3, float>(kp, st, e);
  return false;
}
}  // namespace ss
