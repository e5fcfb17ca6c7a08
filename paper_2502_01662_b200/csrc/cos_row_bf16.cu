// The launch of a run in one, for bf16 logits.
#include "cos_row_launch.cuh"

namespace cosv {

template cudaError_t row_launch<COS_DTYPE_BF16>(const KParams&, int, int, cudaStream_t);

int row_clusters(int parts) {
  KernelFn fn = cos_row_kernel<COS_DTYPE_BF16, kEnsembleSample, 2, true, 0>;
  const int smem = 120 * 1024;  // (more than half of a multiprocessor's: one block on each)
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(static_cast<unsigned>(parts), 1, 1);
  lc.blockDim = dim3(kRowThreads, 1, 1);
  lc.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = static_cast<unsigned>(parts);
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  int n = 0;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
      cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, fn, &lc) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

}  // namespace cosv
