// tbn_conv_igemm_tma64.cu -- the 64-channel TMA variants of the implicit-GEMM
// convolution kernel (every pool width and epilogue store, with and without
// the fused quantization prologue), compiled apart from the host dispatch.
#include "tbn_conv_igemm.cuh"

namespace tbn {

tbn_status launch_igemm_tma64(const ConvProblem& p, const TilePlan& t, IgArgs& a, int pw,
                              bool tma_store, bool fuse, cudaStream_t s) {
  if (fuse)
    return tma_store ? launch_pool<kModeTma64, true, true>(p, t, a, pw, s)
                     : launch_pool<kModeTma64, false, true>(p, t, a, pw, s);
  return tma_store ? launch_pool<kModeTma64, true, false>(p, t, a, pw, s)
                   : launch_pool<kModeTma64, false, false>(p, t, a, pw, s);
}

// Asked of the driver once per process (one process drives one GPU).  Every
// TMA mode has this kernel's threads and shared memory.
int igemm_max_clusters(int size) {
  static std::once_flag once;
  static int fit[kMaxCluster + 1] = {};
  std::call_once(once, [] {
    auto kern = conv_igemm_kernel<kModeTma64, 0, false, false>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) !=
        cudaSuccess) {
      cudaGetLastError();
      return;
    }
    for (int c = 2; c <= kMaxCluster; ++c) {
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(static_cast<unsigned>(c));
      cfg.blockDim = dim3(threads_for<kModeTma64>());
      cfg.dynamicSmemBytes = smem_bytes_for(kModeTma64, 0, 0);
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = static_cast<unsigned>(c);
      attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      if (cudaOccupancyMaxActiveClusters(&fit[c], kern, &cfg) != cudaSuccess) {
        fit[c] = 0;
        cudaGetLastError();
      }
    }
  });
  return size >= 2 && size <= kMaxCluster ? fit[size] : 0;
}

}  // namespace tbn
