// The launches for f32 logits.
#include "cos_launch.cuh"

namespace cosv {

template cudaError_t stream_launch<COS_DTYPE_F32>(const KParams&, int, int, cudaStream_t);
template cudaError_t decide_launch<COS_DTYPE_F32>(const KParams&, int, cudaStream_t);
template cudaError_t mask_launch<COS_DTYPE_F32>(const KParams&, int, cudaStream_t);
template cudaError_t draw_launch<COS_DTYPE_F32>(const KParams&, bool, int, int, int, cudaStream_t);
template cudaError_t dump_launch<COS_DTYPE_F32>(const KParams&, int, cudaStream_t);

}  // namespace cosv
