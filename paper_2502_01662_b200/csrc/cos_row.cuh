// A whole run in one launch, a cluster of blocks a row: for runs whose rows have their places on the device side by side.
#ifndef COS_ROW_CUH
#define COS_ROW_CUH

#include "cos_draw.cuh"
#include "cos_launch.h"

namespace cosv {

// Split: a row's positions are one line of vectors as in cos_stream_kernel, cut into shares for the warps of the row's cluster, which go
// on with the decisions and the drawing sweep of cos_draw_kernel behind a barrier of the cluster where that waits for a launch.  With a
// plausibility mask the warps first look for the gating model's largest logits in the same shares, behind one barrier more.
// What bounds it: the same chain of latencies, without the ends and beginnings of launches (and what they cost on the host: 2.5 us each),
// but with no more multiprocessors for a row than a cluster has; so it is taken by the rule at plan_row.
// 512 threads: 128 registers, which the sweeps of four models need, and one block on a multiprocessor.

// The largest logits of the gating model, from which the plausibility thresholds follow: a share's part of the positions.
template <int DT, bool AL>
__device__ __forceinline__ void row_mask_share(const KParams& p, int b, int share) {
  constexpr int U = kStreamDepth;
  const int lane = threadIdx.x & 31;
  const VecRange whole = whole_vectors<DT, AL>(p.V);
  for (long long x = worker_lo(p, share), end = worker_lo(p, share + 1); x < end;) {
    const int j = line_div(x, p.st_nv, p.st_inv_nv);
    const int o0 = static_cast<int>(x - static_cast<long long>(j) * p.st_nv);
    const int o1 = end - x < p.st_nv - o0 ? o0 + static_cast<int>(end - x) : p.st_nv;
    x += o1 - o0;
    const char* row = reinterpret_cast<const char*>(p.logits) +
                      (p.mask_model * p.s_model + static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
    float best = -INFINITY;
    const int v1 = whole.lo + o1 < whole.hi ? whole.lo + o1 : whole.hi;
    for (int v = whole.lo + o0 + lane; v < v1; v += U * 32) {
      uint4 raw[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        raw[u] = neg_inf_vector<DT>();
        if (v + u * 32 < v1) raw[u] = load_whole<DT, AL>(row, v + u * 32);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) best = max_nan(best, vector_max<DT, false>(raw[u]));
    }
    if (o1 == p.st_nv) {
      const int e = ragged_entry(ragged_of<DT, AL>(p.V), p.V, lane);
      if (e >= 0) best = max_nan(best, Elem<DT>::load1(row, e));
    }
    const unsigned bits = (best != best) ? 0x7fc00000u : __float_as_uint(best);
    const unsigned top = __reduce_max_sync(0xffffffffu, bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u));
    if (lane == 0) atomicMax(&p.mask_key[b * p.P + j], top);
  }
}

// One of the row's st_warps shares (see cos_stream_kernel).
template <int DT, int MODE, bool AL, bool PAIR, bool MASKED>
__device__ __forceinline__ void row_share(const KParams& p, int b, int w, bool& waited) {
  constexpr bool kEns = (MODE == kEnsembleSample || MODE == kEnsembleGreedy);
  const int slots = record_slots<MODE>(p);
  int share = w, i0 = 0, i1 = p.n;
  if (kEns && p.st_split) {
    const int row = w / p.st_split, unit = row / p.n;
    share = unit * p.st_split + w - row * p.st_split;
    i0 = row - unit * p.n;
    i1 = i0 + 1;
  }
  int4* const recs = p.st_rec + static_cast<size_t>(b) * (p.P + p.st_row) * slots;
  for (long long x = worker_lo(p, share), end = worker_lo(p, share + 1); x < end;) {
    const int j = line_div(x, p.st_nv, p.st_inv_nv);
    const int o0 = static_cast<int>(x - static_cast<long long>(j) * p.st_nv);
    const int o1 = end - x < p.st_nv - o0 ? o0 + static_cast<int>(end - x) : p.st_nv;
    x += o1 - o0;
    const char* base = reinterpret_cast<const char*>(p.logits) +
                       (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
    int pis = 0;
    float thr = -INFINITY;
    if (!kEns) {
      const int pi = proposer_of(p, b, j);
      pis = (pi >= 0 && pi < p.n) ? pi : 0;
      if (MASKED) thr = mask_bound(p, __ldcg(&p.mask_key[b * p.P + j]));
    }
    sweep_part<DT, MODE, AL, PAIR, MASKED>(p, base, o0, o1, i0, i1, pis, thr, recs + (j + share) * slots, waited);
  }
}

// FORM: logit level: bit 0: two models, bit 1: with a mask.  Ensembles: 0.
template <int DT, int MODE, int NCH, bool AL, int FORM>
__global__ void __launch_bounds__(kRowThreads, 1) cos_row_kernel(const __grid_constant__ KParams p) {
  constexpr bool kSample = (MODE == kEnsembleSample || MODE == kLogitSample), kEns = (MODE == kEnsembleSample || MODE == kEnsembleGreedy);
  constexpr bool kPair = (FORM & 1) != 0, kMasked = (FORM & 2) != 0;
  using SH = DrawShared<NCH, kRowParts, kRowSums>;
  extern __shared__ __align__(16) unsigned char row_smem_raw[];
  SH& sh = *reinterpret_cast<SH*>(row_smem_raw);
  double* slots = reinterpret_cast<double*>(row_smem_raw + sizeof(SH));
  RowShared& rs = *reinterpret_cast<RowShared*>(slots);
  double* acc = slots + threadIdx.x;
  const int b = blockIdx.x / p.draw_parts, rank = blockIdx.x % p.draw_parts, nw = blockDim.x >> 5, warp = threadIdx.x >> 5;
  if (kSample) fill_const<DT>(p, sh.kc);
  // Where the caller promises that the inputs are not what the kernel ahead writes, a warp waits for that one only before it writes itself;
  // the promise does not cover an offset in device memory.  Nor does it cover what may run beside the kernel ahead, if that let this one
  // start early: so the call behind may start only when every block of this one has waited.
  // (With a mask the promise is not taken; left open to the compiler it costs the masked sweep 4 to 8 %: 60 rows of 5 x 2 x 64000 46.3 us and 43.1.)
  const bool settled = !kMasked && p.inputs_settled != 0 && p.off_dev == nullptr;
  bool waited = !settled;
  if (!settled) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  const TilePlan t = tile_plan<MODE>(p);
  const TileInputs in = tile_inputs<DT, MODE>(p, t, b, 0);
  if (kMasked) {
    for (int w = rank * nw + warp; w < p.st_warps; w += p.draw_parts * nw) row_mask_share<DT, AL>(p, b, w);
    cluster_arrive();
    cluster_wait();
  }
  for (int w = rank * nw + warp; w < p.st_warps; w += p.draw_parts * nw) row_share<DT, MODE, AL, kPair, kMasked>(p, b, w, waited);
  if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
  if (settled) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cluster_arrive();  // (the records of this block are there, and its shared memory may be written to)
  if (kSample) {
    if (!decide_unit_to_draw<DT, kEns, NCH>(p, sh, rs, t, in, b, -1, rank, [] { cluster_wait(); })) return;
    __syncthreads();
    draw_sweep<DT, kEns, NCH, AL, FORM>(p, sh, rank * nw + warp, p.draw_parts * nw, acc);
    cluster_arrive();
    cluster_wait();
    if (rank == 0) {
      __syncthreads();
      locate<DT, kEns, NCH, AL, FORM>(p, sh, acc);
    }
  } else {
    cluster_wait();
    if (rank == 0) decide_greedy<DT, MODE>(p, rs, t, in, b, [] {});
  }
}

}  // namespace cosv

#endif  // COS_ROW_CUH
