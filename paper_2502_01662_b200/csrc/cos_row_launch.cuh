// The launch of a run in one, for one element type (each is compiled in a unit of its own: cos_row_bf16.cu, cos_row_f16.cu,
// cos_row_f32.cu).
#ifndef COS_ROW_LAUNCH_CUH
#define COS_ROW_LAUNCH_CUH

#include "cos_launch.cuh"
#include "cos_row.cuh"

namespace cosv {

template <int DT, int MODE, bool AL>
KernelFn row_logit_kernel_of(bool pair, bool masked) {
  if (pair) return masked ? cos_row_kernel<DT, MODE, 2, AL, 3> : cos_row_kernel<DT, MODE, 2, AL, 1>;
  return masked ? cos_row_kernel<DT, MODE, 2, AL, 2> : cos_row_kernel<DT, MODE, 2, AL, 0>;
}
template <int DT, bool AL>
KernelFn row_kernel_of(int mode, int channels, bool pair, bool masked) {
  switch (mode) {
    case kEnsembleSample: return channels == 2 ? cos_row_kernel<DT, kEnsembleSample, 2, AL, 0> : cos_row_kernel<DT, kEnsembleSample, 4, AL, 0>;
    case kEnsembleGreedy: return cos_row_kernel<DT, kEnsembleGreedy, 2, AL, 0>;
    case kLogitSample: return row_logit_kernel_of<DT, kLogitSample, AL>(pair, masked);
    default: return row_logit_kernel_of<DT, kLogitGreedy, AL>(pair, masked);
  }
}

template <int DT>
cudaError_t row_launch(const KParams& p, int mode, int channels, cudaStream_t stream) {
  const bool pair = p.n == 2, masked = p.mask_model >= 0;
  KernelFn fn = p.vec_ok ? row_kernel_of<DT, true>(mode, channels, pair, masked) : row_kernel_of<DT, false>(mode, channels, pair, masked);
  const size_t slow = 2 * channels * kRowThreads * sizeof(double);  // (the decisions come first, in the same place)
  const size_t smem = (channels == 4 ? sizeof(DrawShared<4, kRowParts, kRowSums>) : sizeof(DrawShared<2, kRowParts, kRowSums>)) +
                      (slow > sizeof(RowShared) ? slow : sizeof(RowShared));
  cudaError_t e = cudaSuccess;
  if (smem > 48 * 1024) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e == cudaSuccess && p.draw_parts > 8) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  return launch(fn, p, p.B * p.draw_parts, kRowThreads, smem, stream, p.draw_parts);
}

}  // namespace cosv

#endif  // COS_ROW_LAUNCH_CUH
