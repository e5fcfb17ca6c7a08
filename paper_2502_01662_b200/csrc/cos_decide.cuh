// Decisions from the records of a streaming launch: accept tests of a row's positions (Eq. 6), the first rejection and the
// row's outputs (Sec. 3.1).
#ifndef COS_DECIDE_CUH
#define COS_DECIDE_CUH

#include "cos_stream.cuh"

namespace cosv {

// A block decides a whole row: a few lanes merge the records of one (position, slot) pair each, then one warp goes on, a lane taking
// the accept test of a position, a ballot finding the first rejection.  Every block of a row does it for itself (the records of a
// row are a few KB, read from L2), which costs the device nothing that it would use otherwise, and no word has to travel between
// blocks; one of them writes the outputs.
// What bounds it: a chain of latencies, the same the second time that a block goes through it (so not of instructions fetched for the first
// time).  So what it needs of the inputs (drafts, proposers, the logits at the drafts, random words) is there before it waits for the
// streaming launch to end, nothing is read from global memory after the records, and the
// lane of the position to be drawn has all that is needed to draw it.  (With what follows in the drawing launch, device time of a call:
// one row of 5 x 2 x 32000 fp32 14.8 us before and 12.7 now, 32 rows of 6 x 2 x 32000 bf16 25.0 and 22.6.)
constexpr int kTile = 16;  // positions decided at a time

struct PairStats {  // one softmax of a position
  double p;    // probability of the draft token; NaN where the statistics are of no use
  double inv;  // one over the normaliser
  double s;
  float ref, thr;
};
struct RowShared {
  union {
    PairStats pair[kTile][COS_MAX_MODELS];  // sampling
    Finish fin[kTile];                      // greedy
  };
  int a;             // the row's first rejected position, or gamma; -1 until it is known
  int cand;          // greedy: the token there
  float prob;        // greedy: the bonus token's probability
  unsigned status;   // greedy: status bits up to there
  int draft[kTile];  // the draft tokens of the tile
};

// What the merge and the accept tests of a tile need of the inputs, asked for before the records are there.
struct TileInputs {
  RecordRange range;  // the thread's pair
  int at, pair_pi;    // its draft token and proposer
  DraftLogit d;       // (tile_logits)
  int draft, pi;      // the lane's position
  unsigned word0, word1;
};
// A load that stays where it is, before what takes long.
__device__ __forceinline__ int load_now(const int* at) {
  int v;
  asm volatile("ld.global.nc.s32 %0, [%1];" : "=r"(v) : "l"(at));
  return v;
}
__device__ __forceinline__ int proposer_now(const KParams& p, int b, int j) {  // (see proposer_of)
  return j == p.gamma && p.bonus_model >= 0 ? p.bonus_model : load_now(p.proposer + (p.per_pos ? b * p.P + j : b));
}
struct TilePlan {  // pairs of (position, slot) and the lanes that share one: as many as the block has to spare (a thread for each at least)
  int lg, pos, slot, sub;
};
template <int MODE>
__device__ __forceinline__ TilePlan tile_plan(const KParams& p) {
  const int slots = record_slots<MODE>(p), pairs = (p.P < kTile ? p.P : kTile) * slots;
  TilePlan t;
  t.lg = 5;
#pragma unroll 1
  while (pairs << t.lg > blockDim.x) --t.lg;
  const int mine = threadIdx.x >> t.lg;
  t.sub = threadIdx.x & ((1 << t.lg) - 1);
  t.pos = (mine * p.slot_inv) >> 16;
  t.slot = mine - t.pos * slots;
  return t;
}
template <int DT, int MODE>
__device__ __forceinline__ TileInputs tile_inputs(const KParams& p, const TilePlan& t, int b, int j0) {
  constexpr bool kSample = (MODE == kEnsembleSample || MODE == kLogitSample);
  const int count = p.P - j0 < kTile ? p.P - j0 : kTile;
  TileInputs in;
  in.d = {0.0, 0.f};
  in.range = {nullptr, 0};
  in.at = -1;
  in.pair_pi = in.draft = in.pi = 0;
  const bool mine = kSample && t.pos < count && t.sub == 0 && j0 + t.pos < p.gamma;
  if (mine) {
    in.at = load_now(p.drafts + b * p.gamma + j0 + t.pos);
    if (MODE == kLogitSample) in.pair_pi = proposer_now(p, b, j0 + t.pos);
  }
  const int j = j0 + threadIdx.x;
  if (threadIdx.x < count) {
    if (j < p.gamma) in.draft = load_now(p.drafts + b * p.gamma + j);
    in.pi = proposer_now(p, b, j);
  }
  if (t.pos < count) in.range = records_of<MODE>(p, b, j0 + t.pos);
  unsigned rnd[4] = {0u, 0u, 0u, 0u};
  if (threadIdx.x < count)
    philox4x32_10(static_cast<unsigned>(p.row_base + b), static_cast<unsigned>(j), offset_lo(p), offset_hi(p), p.seed_lo, p.seed_hi, rnd);
  in.word0 = rnd[0];
  in.word1 = rnd[1];
  asm volatile("" : "+r"(in.word0), "+r"(in.word1), "+l"(in.range.first), "+r"(in.range.count));  // (now, not where it is used)
  return in;
}
// The logits at the draft tokens, of tile_inputs.
template <int DT, int MODE>
__device__ __forceinline__ void tile_logits(const KParams& p, const TilePlan& t, int b, int j0, TileInputs& in) {
  if (MODE != kEnsembleSample && MODE != kLogitSample) return;
  const char* base = reinterpret_cast<const char*>(p.logits) +
                     (static_cast<long long>(b) * p.s_row + static_cast<long long>(j0 + t.pos) * p.s_pos) * Elem<DT>::bytes;
  if (in.at >= p.V) in.at = -1;
  in.d = draft_logit<DT, MODE>(p, base, t.slot, (in.pair_pi >= 0 && in.pair_pi < p.n) ? in.pair_pi : 0, in.at);
  asm volatile("" : "+d"(in.d.x), "+f"(in.d.gate));
}

// Decide row b, sampling.  `want` >= 0: a position whose statistics the block needs, whatever the first rejection; otherwise the first
// rejected position is what it needs.  `in`: the inputs of the first tile; `ready()` waits for the records.  `keep(stats, j, proposer,
// word, accepted, drawable)` is called by one thread of the first warp with that position's merged statistics, its proposer and the
// random word its token is drawn with.  `writes_row(a)` / `writes_unit(j)`: whether this block writes the row's outputs and a
// position's optional ones.  `AT`: see merge_slot.
template <int DT, int MODE, int AT, typename R, typename K, typename WR, typename WU>
__device__ __forceinline__ void decide_sampled(const KParams& p, RowShared& sh, const TilePlan& t, TileInputs in, int b, int want, R ready, K keep,
                                               WR writes_row, WU writes_unit) {
  constexpr bool kEns = (MODE == kEnsembleSample);
  const int tid = threadIdx.x, lane = tid & 31;
  const int slots = record_slots<MODE>(p);
  const bool optional = p.diag != nullptr || p.keep_stats || p.lse != nullptr;
  int a = -1, drawable = 0;  // (of the first warp)
  unsigned status = 0u;
#pragma unroll 1
  for (int j0 = 0; j0 < p.P; j0 += kTile) {
    const int count = p.P - j0 < kTile ? p.P - j0 : kTile;
    if (j0 > 0) in = tile_inputs<DT, MODE>(p, t, b, j0);
    if (tid < count) sh.draft[tid] = in.draft;
    tile_logits<DT, MODE>(p, t, b, j0, in);
    if (j0 == 0) ready();
    {
      const Merged m = merge_slot<MODE, AT>(p, in.range, t.slot, 1 << t.lg, t.sub);
      if (t.pos < count && t.sub == 0) {
        PairStats o;
        o.s = m.soft.s;
        o.ref = m.soft.ref;
        o.thr = m.thr;
        o.inv = 1.0 / m.soft.s;
        o.p = draft_probability<MODE>(p, in.d, t.slot, in.at, m.thr, m.soft, o.inv);
        sh.pair[t.pos][t.slot] = o;
      }
    }
    __syncthreads();
    if (tid < 32) {
      const int j = j0 + lane;
      const bool is_bonus = j == p.gamma, pi_ok = in.pi >= 0 && in.pi < p.n, draft_ok = is_bonus || (in.draft >= 0 && in.draft < p.V);
      const PairStats* f = sh.pair[lane < count ? lane : 0];
      double r_d = 0.0;
      const double q_d = f[kEns ? (pi_ok ? in.pi : 0) : 0].p;
      if (kEns) {
#pragma unroll 1
        for (int k = 0; k < p.n; ++k) r_d += p.w64[k] * f[k].p;
      } else {
        r_d = f[1].p;
      }
      const bool finite = pi_ok && r_d == r_d && q_d == q_d, tested = finite && !is_bonus && draft_ok;
      const bool accept = tested && accepts(word_to_uniform(in.word0), r_d, q_d);
      const unsigned stops = __ballot_sync(0xffffffffu, lane < count && !accept);  // (the bonus position accepts nothing)
      const bool known = a >= 0;
      if (!known && stops) a = j0 + __ffs(stops) - 1;
      const int asked = want >= 0 ? want : a;
      if (j == asked && lane < count) keep(f, j, in.pi, in.word1, accept ? 1 : 0, finite ? 1 : 0);
      const unsigned own = !finite ? static_cast<unsigned>(COS_ROW_NONFINITE)
                                   : (!draft_ok ? static_cast<unsigned>(COS_ROW_BAD_DRAFT)
                                                : (tested && !(q_d > 0.0) ? static_cast<unsigned>(COS_ROW_Q_ZERO) : 0u));
      if (!known) status |= __reduce_or_sync(0xffffffffu, lane < count && (a < 0 || j <= a) ? own : 0u);
      if (!known && a >= 0) drawable = __shfl_sync(0xffffffffu, finite ? 1 : 0, a - j0);
      if (lane == 0) sh.a = a;
      if (optional && lane < count && writes_unit(j)) {
        const int uidx = b * p.P + j;
        if (p.diag) {
          const float nan = __int_as_float(0x7fc00000);
          float* o = p.diag + static_cast<long long>(uidx) * 4;
          o[0] = !tested ? nan : (q_d > 0.0 ? static_cast<float>(r_d / q_d) : (r_d > 0.0 ? INFINITY : 0.f));
          o[1] = tested ? static_cast<float>(r_d) : nan;
          o[2] = tested ? static_cast<float>(q_d) : nan;
          o[3] = nan;
        }
#pragma unroll 1
        for (int k = 0; k < slots; ++k) {
          if (p.lse) {  // ln sum_x exp(l(x) / T) = (ref + log2 s) ln 2
            SoftPart part;
            part.s = f[k].s;
            part.ref = f[k].ref;
            p.lse[static_cast<long long>(uidx) * slots + k] = log_sum_exp(part, finite);
          }
          if (p.keep_stats) {
            p.ustats[uidx].s[k] = f[k].s;
            p.ustats[uidx].ref[k] = f[k].ref;
            p.ustats[uidx].thr32 = f[k].thr;
          }
        }
        if (p.keep_stats) p.unit_res[uidx] = make_int4(accept ? 1 : 0, static_cast<int>(own), -1, finite ? 1 : 0);
      }
      if (!kEns && p.mask_model >= 0 && lane < count && writes_unit(j)) p.mask_key[b * p.P + j] = 0u;  // ready for the next run
    }
    __syncthreads();
    const int first = sh.a;
    if (first >= 0 && (want < 0 || want < j0 + count) && !optional && p.mask_model < 0) break;
    if (j0 + kTile < p.P) __syncthreads();  // the tile is about to be overwritten
  }
  if (tid < 32 && writes_row(a)) {
#pragma unroll 1
    for (int k = lane; k < p.P; k += 32)
      p.out_tokens[static_cast<long long>(b) * p.P + k] = k < a ? (p.P <= kTile ? sh.draft[k] : p.drafts[b * p.gamma + k]) : -1;
    if (lane == 0) {
      p.accept_count[b] = a;
      p.row_status[b] = status;
      if (p.bonus_prob != nullptr) p.bonus_prob[b] = __int_as_float(0x7fc00000);
      if (p.keep_stats) p.row_draw[b] = drawable ? a : -1;
    }
  }
}

// The same for greedy runs, whose tokens come out of the decisions.
template <int DT, int MODE, typename R>
__device__ __forceinline__ void decide_greedy(const KParams& p, RowShared& sh, const TilePlan& t, TileInputs in, int b, R ready) {
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
  const int slots = record_slots<MODE>(p);
  const bool optional = p.diag != nullptr || p.keep_stats || p.lse != nullptr;
  if (tid == 0) {
    sh.a = -1;
    sh.status = 0u;
  }
#pragma unroll 1
  for (int j0 = 0; j0 < p.P; j0 += kTile) {
    const int count = p.P - j0 < kTile ? p.P - j0 : kTile;
    if (j0 > 0) in = tile_inputs<DT, MODE>(p, t, b, j0);
    if (tid < count) sh.draft[tid] = in.draft;
    if (j0 == 0) ready();
    {
      const Merged m = merge_slot<MODE, 8>(p, in.range, t.slot, 1 << t.lg, t.sub);
      if (t.pos < count && t.sub == 0) {
        Finish& f = sh.fin[t.pos];
        f.farg[t.slot] = m.arg;
        if (t.slot == slots - 1) f.thr = m.thr;
      }
    }
    __syncthreads();
    if (tid < 32) {
      Decision& dec = sh.fin[lane < count ? lane : 0].dec;
      int accept = 0;
      unsigned own = 0u;
      if (lane < count) {
        const bool is_bonus = (j0 + lane == p.gamma);
        const bool draft_ok = is_bonus || (in.draft >= 0 && in.draft < p.V);
        const bool pi_ok = (in.pi >= 0 && in.pi < p.n);
        decide_unit<DT, MODE>(p, sh.fin[lane], dec, word_to_uniform(in.word0), word_to_uniform(in.word1), is_bonus, in.draft, draft_ok, in.pi, pi_ok,
                              pi_ok ? in.pi : 0);
        accept = dec.accept;
        own = static_cast<unsigned>(dec.status);
      }
      const int a = sh.a;
      __syncwarp();
      if (a < 0) {
        const unsigned stops = __ballot_sync(0xffffffffu, lane < count && (!accept || j0 + lane == p.gamma));
        const int k = stops ? __ffs(stops) - 1 : count - 1;
        const unsigned st = __reduce_or_sync(0xffffffffu, lane <= k && lane < count ? own : 0u);
        if (lane == k) {
          sh.status |= st;
          sh.a = stops ? j0 + k : -1;
          sh.cand = dec.cand;
          sh.prob = static_cast<float>(dec.prob);
        }
      }
    }
    __syncthreads();
    const int a = sh.a;
    if (optional) {
#pragma unroll 1
      for (int k = tid; k < count; k += T) {
        const int uidx = b * p.P + j0 + k;
        const Finish& f = sh.fin[k];
        if (p.diag) {
          float* d = p.diag + static_cast<long long>(uidx) * 4;
          d[0] = static_cast<float>(f.dec.ratio);
          d[1] = static_cast<float>(f.dec.r_d);
          d[2] = static_cast<float>(f.dec.q_d);
          d[3] = static_cast<float>(f.dec.S);
        }
        if (p.lse) {
#pragma unroll 1
          for (int i = 0; i < slots; ++i) p.lse[static_cast<long long>(uidx) * slots + i] = __int_as_float(0x7fc00000);
        }
        if (p.keep_stats) {  // the atoms of r, for the test hook
          UnitStats& st = p.ustats[uidx];
          st.pad[0] = (f.dec.status & COS_ROW_NONFINITE) ? -1 : f.dec.natoms;
#pragma unroll 1
          for (int i = 0; i < f.dec.natoms; ++i) {
            st.s[i] = f.dec.atom_mass[i];
            st.ref[i] = __int_as_float(f.dec.atom_tok[i]);
          }
          p.unit_res[uidx] = make_int4(f.dec.accept, f.dec.status, f.dec.cand, f.dec.drawable);
        }
      }
    }
    if (MODE == kLogitGreedy) {
#pragma unroll 1
      for (int k = p.mask_model >= 0 ? tid : count; k < count; k += T) p.mask_key[b * p.P + j0 + k] = 0u;  // ready for the next run
    }
    if (a >= 0 && !optional && p.mask_model < 0) break;
    __syncthreads();  // the tile is about to be overwritten
  }
  const int a = sh.a;
#pragma unroll 1
  for (int k = tid; k < p.P; k += T)
    p.out_tokens[static_cast<long long>(b) * p.P + k] = k < a ? (p.P <= kTile ? sh.draft[k] : p.drafts[b * p.gamma + k]) : (k == a ? sh.cand : -1);
  if (tid == 0) {
    p.accept_count[b] = a;
    p.row_status[b] = sh.status;
    if (p.bonus_prob != nullptr) p.bonus_prob[b] = (a == p.gamma && sh.cand >= 0) ? sh.prob : __int_as_float(0x7fc00000);
  }
}

// The decisions in a launch of their own, one block per row: greedy runs have nothing to draw; ensembles of one or of more than four
// models draw in the launch after it.
template <int DT, int MODE>
__global__ void __launch_bounds__(128) cos_decide_kernel(const __grid_constant__ KParams p) {
  __shared__ RowShared sh;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const TilePlan t = tile_plan<MODE>(p);
  const TileInputs in = tile_inputs<DT, MODE>(p, t, blockIdx.x, 0);
  auto ready = [] { asm volatile("griddepcontrol.wait;" ::: "memory"); };
  if (MODE == kEnsembleSample)
    decide_sampled<DT, MODE, 8>(p, sh, t, in, blockIdx.x, -1, ready, [](const PairStats*, int, int, unsigned, int, int) {}, [](int) { return true; },
                             [](int) { return true; });
  else
    decide_greedy<DT, MODE>(p, sh, t, in, blockIdx.x, ready);
}

}  // namespace cosv

#endif  // COS_DECIDE_CUH
