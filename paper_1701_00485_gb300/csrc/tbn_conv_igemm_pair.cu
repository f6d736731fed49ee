// tbn_conv_igemm_pair.cu -- the tap-pair variants of the implicit-GEMM
// convolution kernel (64 m + 32 channels, wide tiles; every pool width and
// epilogue store, with and without the fused quantization prologue), compiled
// apart from the host dispatch.
#include "tbn_conv_igemm.cuh"

namespace tbn {

tbn_status launch_igemm_tappair(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw,
                                bool tma_store, bool fuse, cudaStream_t s) {
  if (fuse)
    return tma_store ? launch_pool<kModeTapPair, true, true>(p, t, a, pw, s)
                     : launch_pool<kModeTapPair, false, true>(p, t, a, pw, s);
  return tma_store ? launch_pool<kModeTapPair, true, false>(p, t, a, pw, s)
                   : launch_pool<kModeTapPair, false, false>(p, t, a, pw, s);
}

}  // namespace tbn
