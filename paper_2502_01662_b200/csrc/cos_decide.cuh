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
// What bounds it: a chain of latencies, and fetching instructions that no other block has run before (5 us from the end of the
// streaming launch to the first load of the drawing sweep).  So what it needs of the inputs (drafts, proposers, the logits at the
// drafts) is asked for before it waits for the streaming launch to end, there is one copy of everything and little is
// unrolled: with fetches in two copies, 64-bit divisions and unrolled cold loops (35 KB instead of 20) it took 11 us.  Going
// through it once on stale records before the wait, to have the instructions at hand, cost 4 to 8 us: the first time is the slow
// one wherever it is.
constexpr int kTile = 16;  // positions decided at a time

struct RowShared {
  Finish fin[kTile];
  int a;            // the row's first rejected position, or gamma; -1 until it is known
  int drawable;     // whether a token can be drawn there
  int cand;         // greedy: the token there
  float prob;       // greedy: the bonus token's probability
  unsigned status;  // status bits up to there
};

// Decide row b.  `want` >= 0: a position whose statistics the block needs, whatever the first rejection; otherwise the first
// rejected position is what it needs.  `keep(fin, j, word, accepted, drawable)` is called by the first warp with that position's
// merged statistics and the random word its token is drawn with.  `writes_row(a)` / `writes_unit(j)`: whether this block writes
// the row's outputs and a position's optional ones.
template <int DT, int MODE, typename K, typename WR, typename WU>
__device__ __forceinline__ void decide_row(const KParams& p, RowShared& sh, int b, int want, K keep, WR writes_row, WU writes_unit) {
  constexpr bool kSample = (MODE == kEnsembleSample || MODE == kLogitSample);
  const int tid = threadIdx.x, lane = tid & 31, T = blockDim.x;
  const int slots = record_slots<MODE>(p);
  const bool optional = p.diag != nullptr || p.keep_stats || p.lse != nullptr;
  // lanes that share a pair: as many as the block has to spare (it has a thread for each at least)
  const int pairs = (p.P < kTile ? p.P : kTile) * slots;
  int lg = 5;
#pragma unroll 1
  while (pairs << lg > T) --lg;
  const int mine = tid >> lg, sub = tid & ((1 << lg) - 1);
  const int pos = (mine * p.slot_inv) >> 16, i = mine - pos * slots;
  const char* row = reinterpret_cast<const char*>(p.logits) + static_cast<long long>(b) * p.s_row * Elem<DT>::bytes;
  if (tid == 0) {
    sh.a = -1;
    sh.status = 0u;
  }
#pragma unroll 1
  for (int j0 = 0; j0 < p.P; j0 += kTile) {
    const int count = p.P - j0 < kTile ? p.P - j0 : kTile;
    const bool live = pos < count;
    // what the merge and the accept test need of the inputs
    DraftLogits d = {0.f, 0.f};
    RecordRange range = {nullptr, 0};
    int at = -1;  // the pair's draft token
    const char* base = row + static_cast<long long>(j0 + pos) * p.s_pos * Elem<DT>::bytes;
    if (live) {
      const int j = j0 + pos;
      range = records_of<MODE>(p, b * p.P + j);
      if (kSample && sub == 0 && j < p.gamma) {
        at = __ldg(p.drafts + b * p.gamma + j);
        if (at >= p.V) at = -1;
        const int pi = (MODE == kLogitSample) ? proposer_of(p, b, j) : 0;
        d = draft_logits<DT, MODE>(p, base, i, (pi >= 0 && pi < p.n) ? pi : 0, at);
      }
    }
    int draft = 0, pi = 0;
    unsigned rnd[4] = {0u, 0u, 0u, 0u};
    if (tid < count) {
      const int j = j0 + tid;
      if (j < p.gamma) draft = __ldg(p.drafts + b * p.gamma + j);
      pi = proposer_of(p, b, j);
      philox4x32_10(static_cast<unsigned>(p.row_base + b), static_cast<unsigned>(j), offset_lo(p), offset_hi(p), p.seed_lo, p.seed_hi, rnd);
    }
    if (j0 == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    {
      const Merged m = merge_slot<MODE>(p, range, i, 1 << lg, sub);
      if (live && sub == 0) {
        Finish& f = sh.fin[pos];
        if (kSample) {
          f.fsoft[i] = m.soft;
          f.inv[i] = 1.0 / m.soft.s;
          f.pdraft[i] = draft_probability<DT, MODE>(p, d, base, i, at, m.thr, m.soft, f.inv[i]);
        } else {
          f.farg[i] = m.arg;
        }
        if (i == slots - 1) f.thr = m.thr;
      }
    }
    __syncthreads();
    if (tid < 32) {
      // (sampling: the decision stays in registers but where somebody asked to see it)
      Decision own;
      own.accept = own.status = own.drawable = 0;
      Decision& dec = kSample || lane >= count ? own : sh.fin[lane].dec;
      if (lane < count) {
        const bool is_bonus = (j0 + lane == p.gamma);
        const bool draft_ok = is_bonus || (draft >= 0 && draft < p.V);
        const bool pi_ok = (pi >= 0 && pi < p.n);
        decide_unit<DT, MODE>(p, sh.fin[lane], dec, word_to_uniform(rnd[0]), word_to_uniform(rnd[1]), is_bonus, draft, draft_ok, pi, pi_ok,
                              pi_ok ? pi : 0);
        if (kSample && optional) sh.fin[lane].dec = dec;
      }
      int a = sh.a;
      __syncwarp();
      if (a < 0) {
        const unsigned stops = __ballot_sync(0xffffffffu, lane < count && (!dec.accept || j0 + lane == p.gamma));
        const int k = stops ? __ffs(stops) - 1 : count - 1;
        const unsigned st = __reduce_or_sync(0xffffffffu, lane <= k && lane < count ? static_cast<unsigned>(dec.status) : 0u);
        if (stops) a = j0 + k;
        if (lane == k) {
          sh.status |= st;
          sh.a = a;
          sh.drawable = dec.drawable;
          if (!kSample) {
            sh.cand = dec.cand;
            sh.prob = static_cast<float>(dec.prob);
          }
        }
      }
      const int asked = want >= 0 ? want : a;
      const int k = asked >= j0 && asked < j0 + count ? asked - j0 : 0;
      const int accepted = __shfl_sync(0xffffffffu, dec.accept, k), drawable = __shfl_sync(0xffffffffu, dec.drawable, k);
      const unsigned word = __shfl_sync(0xffffffffu, rnd[1], k);
      if (asked >= j0 && asked < j0 + count) keep(sh.fin[k], asked, word, accepted, drawable);
    }
    __syncthreads();
    const int a = sh.a;
    const int asked = want >= 0 ? want : a;
    if (optional) {
#pragma unroll 1
      for (int k = tid; k < count; k += T) {
        const int j = j0 + k, uidx = b * p.P + j;
        if (!writes_unit(j)) continue;
        const Finish& f = sh.fin[k];
        if (p.diag) {
          float* d = p.diag + static_cast<long long>(uidx) * 4;
          d[0] = static_cast<float>(f.dec.ratio);
          d[1] = static_cast<float>(f.dec.r_d);
          d[2] = static_cast<float>(f.dec.q_d);
          d[3] = static_cast<float>(f.dec.S);
        }
        if (p.lse) {  // ln sum_x exp(l(x) / T) = (ref + log2 s) ln 2
#pragma unroll 1
          for (int i = 0; i < slots; ++i)
            p.lse[static_cast<long long>(uidx) * slots + i] = log_sum_exp(f.fsoft[i], kSample && !(f.dec.status & COS_ROW_NONFINITE));
        }
        if (p.keep_stats) {
          UnitStats& st = p.ustats[uidx];
          if (kSample) {
#pragma unroll 1
            for (int i = 0; i < slots; ++i) {
              st.s[i] = f.fsoft[i].s;
              st.ref[i] = f.fsoft[i].ref;
            }
            st.thr32 = f.thr;
          } else {  // the atoms of r, for the test hook
            st.pad[0] = (f.dec.status & COS_ROW_NONFINITE) ? -1 : f.dec.natoms;
#pragma unroll 1
            for (int i = 0; i < f.dec.natoms; ++i) {
              st.s[i] = f.dec.atom_mass[i];
              st.ref[i] = __int_as_float(f.dec.atom_tok[i]);
            }
          }
          p.unit_res[uidx] = make_int4(f.dec.accept, f.dec.status, f.dec.cand, f.dec.drawable);
        }
      }
    }
    if (MODE == kLogitSample || MODE == kLogitGreedy) {
#pragma unroll 1
      for (int k = p.mask_model >= 0 ? tid : count; k < count; k += T)
        if (writes_unit(j0 + k)) p.mask_key[b * p.P + j0 + k] = 0u;  // ready for the next run
    }
    if (a >= 0 && asked < j0 + count && !optional && p.mask_model < 0) break;
    __syncthreads();  // the tile is about to be overwritten
  }
  const int a = sh.a;
  if (writes_row(a)) {
#pragma unroll 1
    for (int k = tid; k < p.P; k += T)
      p.out_tokens[static_cast<long long>(b) * p.P + k] = k < a ? p.drafts[b * p.gamma + k] : (k == a && !kSample ? sh.cand : -1);
    if (tid == 0) {
      p.accept_count[b] = a;
      p.row_status[b] = sh.status;
      if (p.bonus_prob != nullptr) p.bonus_prob[b] = (!kSample && a == p.gamma && sh.cand >= 0) ? sh.prob : __int_as_float(0x7fc00000);
      if (kSample && p.keep_stats) p.row_draw[b] = sh.drawable ? a : -1;
    }
  }
}

// The decisions in a launch of their own, one block per row: greedy runs have nothing to draw; ensembles of one or of more than four
// models draw in the launch after it.
template <int DT, int MODE>
__global__ void __launch_bounds__(128) cos_decide_kernel(const __grid_constant__ KParams p) {
  __shared__ RowShared sh;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  decide_row<DT, MODE>(p, sh, blockIdx.x, -1, [](const Finish&, int, unsigned, int, int) {}, [](int) { return true; }, [](int) { return true; });
}

}  // namespace cosv

#endif  // COS_DECIDE_CUH
