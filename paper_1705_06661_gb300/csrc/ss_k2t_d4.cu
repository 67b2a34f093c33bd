// Instantiates the TMA-fed tiled kernel for d = 4 (see ss_k2t.cuh).
#include "ss_k2t.cuh"

namespace ss {

// FP64: 48 KB stages, two per CTA and two CTAs per SM (A[112]^4: 738 us at that time, 560 now; four stages of one
// CTA 869, the same with two groups of eight warps 829: one warp then feeds the whole SM)
bool launch_k2t_d4(const KParams& kp, int ar, cudaStream_t st, cudaError_t* e) {
  if (ar == AR_EXACT && (kp.flags & KF_WHT)) return launch_k2t<4, AR_EXACT_XW, 2, 2, double>(kp, st, e);
  if (ar == AR_F32) return launch_k2t<4, AR_F32, 3, 2, float>(kp, st, e);
  return false;
}
}  // namespace ss
