// Internal interface between the translation units of the library: the launches of a run, one unit per element type.
#ifndef COS_LAUNCH_H
#define COS_LAUNCH_H

#include <cuda_runtime.h>

#include "cos_common.cuh"

namespace cosv {

// The streaming launch (mode: the Mode enum): p.st_warps warps, blocks of `threads` threads; with p.early_exit (p.st_workers blocks) or
// p.use_jobs a form that also decides and publishes.  mask: the launch before it that finds the plausibility threshold of every
// position.  decide: a launch after it that decides the rows (greedy runs, and
// ensembles of one or of more than four models).
template <int DT>
cudaError_t stream_launch(const KParams& p, int mode, int threads, cudaStream_t stream);
template <int DT>
cudaError_t decide_launch(const KParams& p, int mode, cudaStream_t stream);
template <int DT>
cudaError_t mask_launch(const KParams& p, int threads, cudaStream_t stream);
// The drawing launch with `channels` 2, 4 or 8 (logit level: 2) for `units` positions: a cluster of p.draw_parts blocks of `threads`
// threads for each.
template <int DT>
cudaError_t draw_launch(const KParams& p, bool ensemble, int channels, int units, int threads, cudaStream_t stream);
// A run in one launch (cos_row.cuh): a cluster of p.draw_parts blocks for each of the p.B rows.
constexpr int kRowThreads = 512, kRowParts = 16, kRowSums = 2048;  // threads of a block, most blocks of a cluster, chunks times channels
template <int DT>
cudaError_t row_launch(const KParams& p, int mode, int channels, cudaStream_t stream);
// Clusters of `parts` such blocks that the current device holds at once; 0: it takes none.
int row_clusters(int parts);
// Test hook: the combined distribution of every position.
template <int DT>
cudaError_t dump_launch(const KParams& p, int mode, cudaStream_t stream);

}  // namespace cosv

#endif  // COS_LAUNCH_H
