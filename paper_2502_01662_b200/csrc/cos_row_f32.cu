// The launch of a run in one, for fp32 logits.
#include "cos_row_launch.cuh"

namespace cosv {

template cudaError_t row_launch<COS_DTYPE_F32>(const KParams&, int, int, cudaStream_t);

}  // namespace cosv
