// tbn_conv_igemm_pad.cu -- the padded-channel TMA variants of the implicit-GEMM
// convolution kernel (C % 8 == 0 channel counts that are no multiple of 32)
// and its row-pair variant (at most 64 filters), compiled apart from the host
// dispatch.
#include "tbn_conv_igemm.cuh"

namespace tbn {

tbn_status launch_igemm_pad(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw,
                            bool tma_store, cudaStream_t s) {
  return tma_store ? launch_pool<kModeTmaPad, true, false>(p, t, a, pw, s)
                   : launch_pool<kModeTmaPad, false, false>(p, t, a, pw, s);
}

tbn_status launch_igemm_rowpair(const ConvProblem& p, const TilePlan& t, IgArgs& a,
                                cudaStream_t s) {
  return launch_t<kModeRowPair, 0, true, false>(p, t, a, s);
}

}  // namespace tbn
