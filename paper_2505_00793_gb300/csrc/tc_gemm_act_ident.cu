// Activation-epilogue instances of the tcgen05 dual GEMM for ACT_IDENT (forward: bias + phi,
// phi' z' and the derivatives the backward needs), and the backward instance of every
// activation (dz = phi' da, dz' = phi'' z' da + phi' da' from the derivatives the forward stored).
// One translation unit per activation so that the instances compile in parallel.
#include "tc_gemm_impl.cuh"

namespace mf {

cudaError_t tc_gemm_act_ident(const GemmArgs& a, cudaStream_t s, const char** why, int bn,
                              int pair) {
  if (a.epi.mode == EPI_ACT_FWD) return launch_bn<EPI_ACT_FWD, ACT_IDENT>(a, s, why, bn, pair);
  return launch_bn<EPI_ACT_BWD, ACT_IDENT>(a, s, why, bn, pair);
}

}  // namespace mf
