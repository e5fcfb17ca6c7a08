// The launches of one element type (each is compiled in a unit of its own: cos_bf16.cu, cos_f16.cu, cos_f32.cu).
#ifndef COS_LAUNCH_CUH
#define COS_LAUNCH_CUH

#include "cos_draw.cuh"
#include "cos_launch.h"
#include "cos_stream.cuh"

namespace cosv {

using KernelFn = void (*)(const KParams);

template <int DT, bool AL>
KernelFn draw_kernel_of(bool ens, int channels, bool pair, bool masked) {
  if (!ens && pair) return masked ? cos_draw_kernel<DT, false, 2, AL, 3> : cos_draw_kernel<DT, false, 2, AL, 1>;
  if (!ens) return masked ? cos_draw_kernel<DT, false, 2, AL, 2> : cos_draw_kernel<DT, false, 2, AL, 0>;
  if (channels == 2) return cos_draw_kernel<DT, true, 2, AL, 0>;
  return channels == 4 ? cos_draw_kernel<DT, true, 4, AL, 0> : cos_draw_kernel<DT, true, 8, AL, 0>;
}

template <int DT, int MODE, bool AL>
KernelFn logit_kernel_of(bool pair, bool masked) {
  if (pair) return masked ? cos_stream_kernel<DT, MODE, AL, true, true> : cos_stream_kernel<DT, MODE, AL, true, false>;
  return masked ? cos_stream_kernel<DT, MODE, AL, false, true> : cos_stream_kernel<DT, MODE, AL, false, false>;
}

// Shares of an ensemble from this many vectors on are long.  Device time of a call with the short and with the long form, in us: 2376
// vectors (64 rows of 9 positions of 2 x 151936 bf16) 84.5 and 81.8, 1625 (96 rows of 5 of 2 x 128256) 83.1 and 81.1, 1083 (64 of
// them) 53.6 and 53.4, 758 (32 rows of 7 of 4 x 128256) 64.6 and 64.0, 507 (48 rows of 5 of 2 x 80000) 39.6 and 40.4, 288 (32 rows
// of 6 of 2 x 32000) 25.1 and 27.0.
constexpr int kLongShare = 640;

template <int DT, bool AL>
KernelFn stream_kernel_of(int mode, bool pair, bool masked, bool long_share) {
  switch (mode) {
    case kEnsembleSample:
      return long_share ? cos_stream_kernel<DT, kEnsembleSample, AL, true, false> : cos_stream_kernel<DT, kEnsembleSample, AL, false, false>;
    case kEnsembleGreedy: return cos_stream_kernel<DT, kEnsembleGreedy, AL, true, false>;
    case kLogitSample: return logit_kernel_of<DT, kLogitSample, AL>(pair, masked);
    default: return logit_kernel_of<DT, kLogitGreedy, AL>(pair, masked);
  }
}
template <int DT>
KernelFn report_kernel_of(int mode, bool pair, bool long_share) {
  if (mode == kEnsembleSample) return long_share ? cos_report_kernel<DT, kEnsembleSample, true> : cos_report_kernel<DT, kEnsembleSample, false>;
  return pair ? cos_report_kernel<DT, kLogitSample, true> : cos_report_kernel<DT, kLogitSample, false>;
}
template <int DT, bool AL>
KernelFn early_kernel_of(int mode) {
  switch (mode) {
    case kEnsembleSample: return cos_early_kernel<DT, kEnsembleSample, AL>;
    case kEnsembleGreedy: return cos_early_kernel<DT, kEnsembleGreedy, AL>;
    case kLogitSample: return cos_early_kernel<DT, kLogitSample, AL>;
    default: return cos_early_kernel<DT, kLogitGreedy, AL>;
  }
}

// Every launch carries the programmatic-stream-serialisation attribute: its blocks take their places while the kernel
// before it drains, and wait for it before they touch anything.
inline cudaError_t launch(KernelFn fn, const KParams& p, int blocks, int threads, size_t smem, cudaStream_t stream, int cluster = 1) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(static_cast<unsigned>(blocks), 1, 1);
  lc.blockDim = dim3(static_cast<unsigned>(threads), 1, 1);
  lc.dynamicSmemBytes = smem;
  lc.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = static_cast<unsigned>(cluster);
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = cluster > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&lc, fn, p);
}

template <int DT>
cudaError_t stream_launch(const KParams& p, int mode, int threads, cudaStream_t stream) {
  if (p.early_exit) return launch(p.vec_ok ? early_kernel_of<DT, true>(mode) : early_kernel_of<DT, false>(mode), p, p.st_workers, threads, 0, stream);
  const int blocks = (p.st_warps + threads / 32 - 1) / (threads / 32);
  const bool pair = p.n == 2, masked = p.mask_model >= 0, long_share = p.st_share >= kLongShare;
  if (p.use_jobs)  // (aligned rows, no mask)
    return launch(report_kernel_of<DT>(mode, pair, long_share), p, blocks, threads, 0, stream);
  return launch(p.vec_ok ? stream_kernel_of<DT, true>(mode, pair, masked, long_share) : stream_kernel_of<DT, false>(mode, pair, masked, long_share), p,
                blocks, threads, 0, stream);
}

template <int DT>
cudaError_t decide_launch(const KParams& p, int mode, cudaStream_t stream) {
  KernelFn fn = mode == kEnsembleGreedy ? cos_decide_kernel<DT, kEnsembleGreedy>
                                        : (mode == kLogitGreedy ? cos_decide_kernel<DT, kLogitGreedy> : cos_decide_kernel<DT, kEnsembleSample>);
  return launch(fn, p, p.B, 128, 0, stream);
}

template <int DT>
cudaError_t mask_launch(const KParams& p, int threads, cudaStream_t stream) {
  const int blocks = (p.st_warps + threads / 32 - 1) / (threads / 32);
  return launch(p.vec_ok ? cos_mask_kernel<DT, true> : cos_mask_kernel<DT, false>, p, blocks, threads, 0, stream);
}

template <int DT>
cudaError_t draw_launch(const KParams& p, bool ens, int channels, int units, int threads, cudaStream_t stream) {
  const bool pair = p.n == 2, masked = p.mask_model >= 0;
  KernelFn fn = p.vec_ok ? draw_kernel_of<DT, true>(ens, channels, pair, masked) : draw_kernel_of<DT, false>(ens, channels, pair, masked);
  const size_t fixed = channels == 2 ? sizeof(DrawShared<2>) : (channels == 4 ? sizeof(DrawShared<4>) : sizeof(DrawShared<8>));
  static_assert(sizeof(DrawShared<4>) + 8 * 8 * kMaxDrawThreads <= 48 * 1024 && sizeof(DrawShared<8>) + 8 * 16 * 256 <= 48 * 1024,
                "no opt-in for large shared memory is made");
  const size_t slow = 2 * channels * threads * sizeof(double);  // (the decisions come first, in the same place)
  return launch(fn, p, units * p.draw_parts, threads, fixed + (slow > sizeof(RowShared) ? slow : sizeof(RowShared)), stream, p.draw_parts);
}

template <int DT>
cudaError_t dump_launch(const KParams& p, int mode, cudaStream_t stream) {
  const dim3 grid(64, static_cast<unsigned>(p.num_units), 1);
  if (mode == kEnsembleSample || mode == kLogitSample)
    cos_dump_kernel<DT><<<grid, 256, 0, stream>>>(p, mode == kEnsembleSample);
  else
    cos_dump_atoms_kernel<DT><<<grid, 256, 0, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace cosv

#endif  // COS_LAUNCH_CUH
