// The drawing launch of a run at T > 0: one sweep over the vocabulary of every position that needs a token (residual
// resample of Sec. 3.2, bonus token of Sec. 3.1), then the token itself.
#ifndef COS_DRAW_CUH
#define COS_DRAW_CUH

#include "cos_decide.cuh"

namespace cosv {

// A token's mass is max(0, sum_i k_i e_i / Z_i), e_i = 2^(x_i c - ref_i), where the channels i are the models (ensemble)
// or the proposer's and the combined logits (logit level) and the k_i say what is drawn: max(0, r - q), r or q.  The set
// of tokens with a positive mass is decided with the normalisers the streaming launch left (good to 1e-7; a token whose
// sign that could change carries no mass to speak of), products rounded one by one so that equal terms cancel exactly.
// Over that set the mass is linear in the 1/Z_i, so the sweep only adds up e_i over it, next to the refined normalisers.
//
// Split: a position is shared by one cluster of p.draw_parts blocks, its steps (32 lanes x one 16-byte vector of every model)
// dealt out in equal consecutive runs to the cluster's warps; a warp sends one record of sums for each chunk of p.draw_cs steps to
// the shared memory of the cluster's first block, nothing per step.  After one barrier of the cluster that block alone
// adds the records up, finds the chunk that holds the token, then the step, then the token.  The host picks block size and parts so
// that the launch fills the device in one wave (see draw_plan).
// The part behind the sweep is a chain of latencies: bank conflicts, loops that need not be loops and second trips to memory for what is in
// registers are what it can do without (cycles in one row of 5 x 2 x 32000 fp32: chunk 3900 with conflicts and serial searches, 2500
// without; the steps' masses 4000, entries and exponentials of big tokens fetched again; token 1000 to 2000 with a load of its entries).
// Records in global memory and the last block to report (fence and counter) took 5 us longer; two more barriers of the cluster, for all
// blocks to look for the token, 1.
constexpr int kMaxDrawThreads = 512;
constexpr int kMaxDrawWarps = kMaxDrawThreads / 32;
constexpr int kMaxParts = 8;       // blocks of a cluster
constexpr int kMaxSums = 768;      // chunks of a position times channels

// Every thread of the cluster arrives and waits; what was written before, to a peer's shared memory too, is visible after.
__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of a place in this block's shared memory, in the cluster's first block.
__device__ __forceinline__ unsigned at_first(const double* mine) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(static_cast<unsigned>(__cvta_generic_to_shared(mine))));
  return r;
}
__device__ __forceinline__ void store_cluster(unsigned a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

// Sums of N values over the warp at once: lane L ends up with the sum of value (L * N / 32).
template <int N>
__device__ __forceinline__ double warp_sums(double (&v)[N], int lane) {
  int n = N;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    const bool upper = (lane & d) != 0;
    if (n > 1) {
      n >>= 1;
#pragma unroll
      for (int i = 0; i < N / 2; ++i)
        if (i < n) {
          const double give = upper ? v[i] : v[i + n], keep = upper ? v[i + n] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, give, d);
        }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], d);
    }
  }
  return v[0];
}

// Where the sums of chunk c are among the records: a record is left out after every eight, so that lanes that each go through a few
// consecutive chunks read from different banks (without, all 32 from the same two: 2.4 of the 6.1 thousand cycles of the search in 512).
__device__ __forceinline__ int record_at(int c) { return c + (c >> 3); }

// Running total over the lanes of a warp (the first N of them are asked for).  Unrolled: 220 cycles for 32 lanes, in a loop 480.
template <int N>
__device__ __forceinline__ double running_total(double m, int lane) {
#pragma unroll
  for (int d = 1; d < N; d <<= 1) {
    const double o = __shfl_up_sync(0xffffffffu, m, d);
    if (lane >= d) m += o;
  }
  return m;
}

// What the functions that are not inlined need of the parameters, in shared memory: behind a call the parameters are no longer
// operands from the constant bank but loads through a generic address, a trip to L2 for each line of them the first time.
struct DrawConst {
  long long row_step;  // bytes from one model's row to the next
  double cT64, w64[COS_MAX_MODELS];
  float cT, w[COS_MAX_MODELS];
  int n, V, mask_model;
};

template <int DT>
__device__ __forceinline__ void fill_const(const KParams& p, DrawConst& kc) {
  if (threadIdx.x < COS_MAX_MODELS) {
    kc.w[threadIdx.x] = p.w[threadIdx.x];
    kc.w64[threadIdx.x] = p.w64[threadIdx.x];
    if (threadIdx.x == 0) {
      kc.row_step = p.s_model * Elem<DT>::bytes;
      kc.cT64 = p.cT64;
      kc.cT = p.cT;
      kc.n = p.n;
      kc.V = p.V;
      kc.mask_model = p.mask_model;
    }
  }
}

// What a block knows about its position.
template <int NCH>
struct DrawUnit {
  const char* base;      // logits of model 0 at this position
  int b, j, uidx;
  int pis;               // model whose distribution is q
  int law;               // kDrawResidual, kDrawR or kDrawQ
  unsigned word;         // the random word the token is drawn with
  int emit;              // the token drawn here is the row's output (else only the residual mass is wanted)
  int accepted, drawable;
  float thr;             // plausibility threshold
  float nref[NCH], bt[NCH], ct[NCH];  // minus the reference exponents, "big" bounds, k / Z in fp32
  double ck[NCH];                     // k / Z
};

template <bool ENS>
__device__ __forceinline__ double coefficient(const KParams& p, int i, int pis, int law) {  // k_i
  if (ENS) {
    const double sel = (i == pis) ? 1.0 : 0.0;
    return i >= p.n ? 0.0 : (law == kDrawResidual ? p.w64[i] - sel : (law == kDrawQ ? sel : p.w64[i]));
  }
  return (i == 0) ? (law == kDrawResidual ? -1.0 : (law == kDrawQ ? 1.0 : 0.0)) : (law == kDrawQ ? 0.0 : 1.0);
}

// Position `u` of the launch; false when nothing is drawn there.  Same values in every thread.
template <int DT, bool ENS, int NCH>
__device__ __forceinline__ bool load_unit(const KParams& p, int u, DrawUnit<NCH>& d) {
  if (!p.draw_all) {
    d.b = u;
    d.j = __ldcg(&p.row_draw[u]);
    if (d.j < 0) return false;
    d.emit = 1;
  } else {
    const int drafts = p.B * p.gamma;  // every draft position, then the bonus positions
    d.b = u < drafts ? u / p.gamma : u - drafts;
    d.j = u < drafts ? u % p.gamma : p.gamma;
    d.emit = (__ldcg(&p.row_draw[d.b]) == d.j) ? 1 : 0;
    if (d.j == p.gamma && !d.emit) return false;
  }
  d.uidx = d.b * p.P + d.j;
  const UnitStats* st = &p.ustats[d.uidx];
  const int4 res = __ldcg(&p.unit_res[d.uidx]);
  if (!res.w) return false;
  d.accepted = res.x;
  d.drawable = 1;
  const int pi = proposer_of(p, d.b, d.j);
  d.pis = (pi >= 0 && pi < p.n) ? pi : 0;
  d.law = (d.j == p.gamma) ? (p.bonus_model >= 0 ? kDrawQ : kDrawR) : kDrawResidual;
  unsigned rnd[4];
  philox4x32_10(static_cast<unsigned>(p.row_base + d.b), static_cast<unsigned>(d.j), offset_lo(p), offset_hi(p), p.seed_lo, p.seed_hi, rnd);
  d.word = rnd[1];
  d.base = reinterpret_cast<const char*>(p.logits) +
           (static_cast<long long>(d.b) * p.s_row + static_cast<long long>(d.j) * p.s_pos) * Elem<DT>::bytes;
  d.thr = (!ENS && p.mask_model >= 0) ? __ldcg(&st->thr32) : -INFINITY;
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const bool live = i < (ENS ? p.n : 2);
    const double z = live ? __ldcg(&st->s[i]) : 1.0;
    d.nref[i] = live ? -__ldcg(&st->ref[i]) : 0.f;
    d.bt[i] = live ? static_cast<float>(z * kBigShare) : INFINITY;
    d.ck[i] = coefficient<ENS>(p, i, d.pis, d.law) / z;
    d.ct[i] = static_cast<float>(d.ck[i]);
  }
  return true;
}

// A vector of every model (logit level: of the first two).
template <int N>
struct Vectors {
  uint4 r[N];
};
// One entry of a vector, any of them.
template <int DT>
__device__ __forceinline__ float entry_at(const uint4& r, int k) {
  const int w = DT == COS_DTYPE_F32 ? k : k >> 1;
  const unsigned a = (w & 1) ? r.y : r.x, b = (w & 1) ? r.w : r.z, h = (w & 2) ? b : a;
  if (DT == COS_DTYPE_F32) return __uint_as_float(h);
  return entry<DT>(make_uint4((k & 1) ? h >> 16 : h, 0u, 0u, 0u), 0);
}

// fp64 terms of token e, the k-th of the vectors: e_i of every channel (in: whether the token is inside the mask).  For "big" tokens (more
// than 2^-8 of a normaliser) and the bonus token's probability.
template <int DT, bool ENS, int NCH, int FORM>
__device__ __forceinline__ void exact_terms(const DrawConst& p, const DrawUnit<NCH>& u, const Vectors<ENS ? NCH : 2>& v, int e, int k, bool in,
                                            double (&out)[NCH]) {
  double t[NCH];
  if (ENS) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) t[i] = static_cast<double>(entry_at<DT>(v.r[i], k));
  } else {
    const float l0 = entry_at<DT>(v.r[0], k), l1 = entry_at<DT>(v.r[1], k);
    float q = u.pis == 0 ? l0 : l1;
    t[1] = p.w64[0] * static_cast<double>(l0);
    if ((FORM & 1) || p.n >= 2) t[1] = fma(p.w64[1], static_cast<double>(l1), t[1]);
    if (!(FORM & 1)) {
#pragma unroll 1
      for (int i = 2; i < p.n; ++i) {
        const float l = Elem<DT>::load1(u.base + i * p.row_step, e);
        if (i == u.pis) q = l;
        t[1] = fma(p.w64[i], static_cast<double>(l), t[1]);
      }
    }
    t[0] = static_cast<double>(q);
    if (!in) t[1] = -INFINITY;
  }
#pragma unroll(NCH == 2 ? 2 : 1)
  for (int k2 = 0; k2 < NCH; ++k2) {  // (more than two channels: one copy of the exponential)
    double x = 0.0;
#pragma unroll
    for (int i = 0; i < NCH; ++i)
      if (i == k2) x = t[i] * p.cT64 + static_cast<double>(u.nref[i]);
    x = exp2(x);
#pragma unroll
    for (int i = 0; i < NCH; ++i)
      if (i == k2) out[i] = x;
  }
}

// Mass of one token from its fp64 terms under the refined normalisers `inv` = 1 / Z_i.
template <bool ENS, int NCH>
__device__ __forceinline__ double exact_mass(const DrawConst& p, const double* e, const double* inv, int pis, int law) {
  double r = 0.0, q = 0.0;
  if (ENS) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      if (i < p.n) {
        const double pr = e[i] * inv[i];
        r += p.w64[i] * pr;
        if (i == pis) q = pr;
      }
    }
  } else {
    q = e[0] * inv[0];
    r = e[1] * inv[1];
  }
  return law == kDrawR ? r : (law == kDrawQ ? q : fmax(0.0, r - q));
}

// The arguments of the NCH channels for the E tokens of vector v of the row from the vectors of the models; beyond V they are -inf.
template <int DT, bool ENS, int NCH, bool AL, int FORM>
__device__ __forceinline__ void vector_args(const KParams& p, const DrawConst& kc, const DrawUnit<NCH>& u, const Vectors<ENS ? NCH : 2>& rv, int v,
                                            float (&x)[NCH][Elem<DT>::E]) {
  constexpr int E = Elem<DT>::E;
  if (ENS) {
#pragma unroll
    for (int i = 0; i < NCH; ++i)
#pragma unroll
      for (int k = 0; k < E; ++k) x[i][k] = entry<DT>(rv.r[i], k);
  } else {
    const VecRange whole = whole_vectors<DT, AL>(kc.V);
    f32x2 xq[E / 2], cmb[E / 2];
    const LogitWeights lw = {kc.w[0], kc.w[1], u.pis, kc.mask_model, u.thr};
    logit_args<DT, (FORM & 1) != 0, (FORM & 2) != 0>(
        p, lw, rv.r[0], rv.r[1], [&](int i) { return load_vector<DT, AL>(u.base + i * kc.row_step, v, kc.V, whole); }, xq, cmb);
#pragma unroll
    for (int k = 0; k < E; ++k) {  // (beyond V the combination of -inf could be anything)
      x[0][k] = pair_at(xq[k / 2], k);
      x[1][k] = (v * E + k < kc.V) ? pair_at(cmb[k / 2], k) : -INFINITY;
    }
  }
}

// The mass of one big token, the k-th of the vectors.  Out of line.
template <int DT, bool ENS, int NCH, int FORM>
__device__ __noinline__ double big_mass(const DrawConst& p, const DrawUnit<NCH>& u, const double* inv, Vectors<ENS ? NCH : 2> rv, int e, int k, bool in) {
  double d[NCH];
  exact_terms<DT, ENS, NCH, FORM>(p, u, rv, e, k, in, d);
  return exact_mass<ENS, NCH>(p, d, inv, u.pis, u.law);
}

// A lane's vector v that the fast loop left out: one with a big entry, or one at a ragged end of the row (fetched here).  Every entry is added in
// fp64, and a big one's exponential is fp64 too.  The sums go to the lane's slots of `acc`, which are cleared where `first`.  Out of line.  (What the fast loop had
// left out, put off until the end of 32 steps, fetched again and dealt out over the warp entry by entry, took a warp 1400 cycles for every
// step that had any.)
template <int DT, bool ENS, int NCH, bool AL, int FORM>
__device__ __noinline__ void slow_vector(const KParams& p, const DrawConst& kc, const DrawUnit<NCH>& u, Vectors<ENS ? NCH : 2> rv, int v, bool ragged,
                                         bool first, double* acc) {
  constexpr int E = Elem<DT>::E, NR = ENS ? NCH : 2;
  const int T = blockDim.x;
  if (ragged) {
    const VecRange whole = whole_vectors<DT, AL>(kc.V);
#pragma unroll
    for (int i = 0; i < NR; ++i)
      if (i < kc.n) rv.r[i] = load_vector<DT, AL>(u.base + i * kc.row_step, v, kc.V, whole);
  }
  float x[NCH][E];
  vector_args<DT, ENS, NCH, AL, FORM>(p, kc, u, rv, v, x);
  double sz[NCH], sa[NCH];
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    sz[i] = first ? 0.0 : acc[i * T];
    sa[i] = first ? 0.0 : acc[(NCH + i) * T];
  }
  unsigned bigbits = 0u, inbits = 0u;
#pragma unroll
  for (int k = 0; k < E; ++k) {
    float f[NCH], tot = 0.f;
    bool big = false;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      f[i] = ex2_approx(fmaf(x[i][k], kc.cT, u.nref[i]));
      big = big || f[i] > u.bt[i];
      tot = __fadd_rn(tot, __fmul_rn(u.ct[i], f[i]));
    }
    if (big) bigbits |= 1u << k;
    if (ENS || x[1][k] != -INFINITY) inbits |= 1u << k;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      sz[i] += big ? 0.0 : static_cast<double>(f[i]);
      sa[i] += !big && tot > 0.f ? static_cast<double>(f[i]) : 0.0;
    }
  }
#pragma unroll 1
  for (; bigbits; bigbits &= bigbits - 1) {
    const int k = __ffs(bigbits) - 1;
    double d[NCH], t = 0.0;
    exact_terms<DT, ENS, NCH, FORM>(kc, u, rv, v * E + k, k, (inbits >> k) & 1u, d);
#pragma unroll
    for (int i = 0; i < NCH; ++i) t = __dadd_rn(t, __dmul_rn(u.ck[i], d[i]));
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      sz[i] += d[i];
      sa[i] += t > 0.0 ? d[i] : 0.0;
    }
  }
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    acc[i * T] = sz[i];
    acc[(NCH + i) * T] = sa[i];
  }
}

// The vectors of steps c to c + 31 that the fast loop left out (bit k of a lane's `left`: its vector of step c + k), of an ensemble: the warp takes 32
// of their entries at a time, one a lane, and adds them to the lanes' slots of `acc`.  Out of line.
template <int DT, int NCH>
__device__ __noinline__ void slow_entries(const DrawConst& p, const DrawUnit<NCH>& u, int c, unsigned left, double* acc) {
  constexpr int E = Elem<DT>::E, G = 32 / E;
  const int T = blockDim.x, lane = threadIdx.x & 31;
#pragma unroll 1
  for (unsigned any = __reduce_or_sync(0xffffffffu, left); any; any &= any - 1) {
    const int k = __ffs(any) - 1;
    unsigned m = __ballot_sync(0xffffffffu, (left >> k) & 1u);
#pragma unroll 1
    while (m) {
      unsigned t = m;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        if (q < lane / E) t &= t - 1;
        m &= m - 1;
      }
      const int e = t ? ((c + k) * 32 + __ffs(t) - 1) * E + lane % E : p.V;
      if (e >= p.V) continue;
      float x[NCH], tot = 0.f;
      double d[NCH];
      bool big = false;
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        x[i] = -INFINITY;
        if (i < p.n) x[i] = Elem<DT>::load1(u.base + i * p.row_step, e);
      }
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        const float f = ex2_approx(fmaf(x[i], p.cT, u.nref[i]));
        big = big || f > u.bt[i];
        tot = __fadd_rn(tot, __fmul_rn(u.ct[i], f));
        d[i] = static_cast<double>(f);
      }
      bool counts = tot > 0.f;
      if (big) {
#pragma unroll 1
        for (int q = 0; q < NCH; ++q) {  // (one copy of the exponential)
          double v = 0.0;
#pragma unroll
          for (int i = 0; i < NCH; ++i)
            if (i == q) v = static_cast<double>(x[i]) * p.cT64 + static_cast<double>(u.nref[i]);
          v = exp2(v);
#pragma unroll
          for (int i = 0; i < NCH; ++i)
            if (i == q) d[i] = v;
        }
        double t64 = 0.0;
#pragma unroll
        for (int i = 0; i < NCH; ++i) t64 = __dadd_rn(t64, __dmul_rn(u.ck[i], d[i]));
        counts = t64 > 0.0;
      }
#pragma unroll
      for (int i = 0; i < NCH; ++i) {
        acc[i * T] += d[i];
        if (counts) acc[(NCH + i) * T] += d[i];
      }
    }
  }
}

// The steps [s_lo, s_hi) of a position by one warp, in chunks of cs steps: per channel the sum over the tokens with a positive mass,
// for every chunk NCH sums to the records from the rec-th on, and to part the normaliser's share, of all chunks together (both in the cluster's first block).
// The fast loop adds vectors up in fp32, up to 32 of a lane, and leaves those with a big entry, and the ragged ends, to slow_vector.
// What bounds it: instruction issue (counted at logit level, 128 rows of 256000 tokens: 220 instructions a step, 0.55 of the issue
// slots of the average multiprocessor, 0.70 of the busiest).  Loads in flight do not: fetching a step as soon as a place is free,
// so that two are always on their way, gained nothing with two channels and lost 2 to 7 % with four.
template <int DT, bool ENS, int NCH, bool AL, int FORM>
__device__ __forceinline__ void draw_sweep_as(const KParams& p, const DrawConst& kc, const DrawUnit<NCH>& u, int cs, int s_lo, int s_hi, double* acc,
                                              int rec, unsigned recs, unsigned part) {
  constexpr bool PAIR = (FORM & 1) != 0, MASKED = (FORM & 2) != 0;
  constexpr int E = Elem<DT>::E;
  constexpr int NP = NCH / 2;
  constexpr int NR = ENS ? NCH : 2;         // vectors of a step kept in registers
  constexpr int US = (NR == 2) ? 2 : 1;     // steps fetched at a time
  // Slow vectors are finished where they are, which is the shorter chain, or behind the (up to 32) steps that have them, fetched again, where
  // the call in the loop costs registers: by the lane that left them out (`kLater`) or entry by entry over the warp (`kShared`), with nothing live
  // across the call.  Device time in us, where they are / behind, by the lane / over the warp: two models, 16-bit, 60 rows of 5 x 64000 36.9 / 36.7 /
  // 37.4, at temperature 0.7 35.9 / 36.4 / 36.6, 7 rows of 32000 14.9 / 15.1 / 15.2; fp32 46.9 / 44.3 / 44.9; three, 60 rows aligned 57.7 / 52.8 / 54.1,
  // fp32 70.7 / 67.5 / 70.4; four, 66.7 / 61.6 / 63.1; 40 rows of 50001 unaligned of three 54.1 / 52.9 / 51.7 (fp32 72.2 / 71.1 / 70.8), of four 66.3 / 63.8 /
  // 62.6 (fp32 89.4 / 88.6 / 89.7); logit level, 60 rows of two 37.0 / 35.4 / 38.0, of three with a mask 71.9 / 66.0 / 66.4.  Eight channels (five
  // models) by the lane and over the warp: 7 rows of 32000 47.1 / 37.5, 40 of 50001 120.4 / 106.5, fp32 165.9 / 145.5; 60 of 64000 99.8 / 102.1.
  constexpr bool kShared = ENS && (NCH == 8 || (NCH == 4 && !AL)), kLater = kShared || !ENS || NCH == 4 || DT == COS_DTYPE_F32;
  const int lane = threadIdx.x & 31;
  const f32x2 c2 = pack2(p.cT, p.cT);
  const VecRange whole = whole_vectors<DT, AL>(p.V);
  const char* base = u.base;
  const long long row_step = p.s_model * Elem<DT>::bytes;
  f32x2 nref[NP], ct[NP];
  float bt[NCH];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    nref[q] = pack2(u.nref[2 * q], u.nref[2 * q + 1]);
    ct[q] = pack2(u.ct[2 * q], u.ct[2 * q + 1]);
    bt[2 * q] = u.bt[2 * q];
    bt[2 * q + 1] = u.bt[2 * q + 1];
  }
  const LogitWeights lw = logit_weights(p, u.pis, u.thr);
  double all = 0.0;
#pragma unroll 1
  for (int begin = s_lo; begin < s_hi; begin += cs, ++rec) {
    const int end = begin + cs < s_hi ? begin + cs : s_hi;
    bool slow = false;  // (whether the lane's slots hold anything)
    f32x2 zc[NP], ac[NP];
#pragma unroll
    for (int q = 0; q < NP; ++q) zc[q] = ac[q] = pack2(0.f, 0.f);
#pragma unroll 1
    for (int c = begin; c < end; c += 32) {  // (not more in fp32)
      const int ce = c + 32 < end ? c + 32 : end;
      unsigned later = 0u;
#pragma unroll 1
      for (int s = c; s < ce; s += US) {
        Vectors<NR> r[US];
#pragma unroll
        for (int t = 0; t < US; ++t) {
          const int v = (s + t) * 32 + lane;
          const bool in = v >= whole.lo && v < whole.hi;
#pragma unroll
          for (int i = 0; i < NR; ++i) {
            r[t].r[i] = neg_inf_vector<DT>();
            if (in && s + t < ce && i < p.n) r[t].r[i] = load_whole<DT, AL>(base + i * row_step, v);
          }
        }
#pragma unroll
        for (int t = 0; t < US; ++t) {
          f32x2 vz[NP], va[NP];
#pragma unroll
          for (int q = 0; q < NP; ++q) vz[q] = va[q] = pack2(0.f, 0.f);
          if (ENS) {
            // two channels side by side in every packed instruction
#pragma unroll
            for (int k = 0; k < E; ++k) {
              f32x2 e[NP], m[NP];
#pragma unroll
              for (int q = 0; q < NP; ++q) {
                const f32x2 arg = fma2(pack2(entry<DT>(r[t].r[2 * q], k), entry<DT>(r[t].r[2 * q + 1], k)), c2, nref[q]);
                e[q] = pack2(ex2_approx(lo2(arg)), ex2_approx(hi2(arg)));
                vz[q] = add2(vz[q], e[q]);
                m[q] = mul2(ct[q], e[q]);
              }
              float tot = __fadd_rn(lo2(m[0]), hi2(m[0]));
#pragma unroll
              for (int q = 1; q < NP; ++q) tot = __fadd_rn(__fadd_rn(tot, lo2(m[q])), hi2(m[q]));
#pragma unroll
              for (int q = 0; q < NP; ++q) add2_if(va[q], e[q], tot);
            }
          } else {
            // two neighbouring tokens side by side
            f32x2 xq[E / 2], cmb[E / 2];
            const int v = (s + t) * 32 + lane;
            const bool in = v >= whole.lo && v < whole.hi && s + t < ce;
            logit_args<DT, PAIR, MASKED>(p, lw, r[t].r[0], r[t].r[1],
                                         [&](int i) {
                                           uint4 m = neg_inf_vector<DT>();
                                           if (in) m = load_whole<DT, AL>(base + i * row_step, v);
                                           return m;
                                         },
                                         xq, cmb);
            f32x2 zq = pack2(0.f, 0.f), zm = zq;
            float aq = 0.f, am = 0.f;
            const f32x2 nq = pack2(lo2(nref[0]), lo2(nref[0])), nm = pack2(hi2(nref[0]), hi2(nref[0]));
            const f32x2 cq = pack2(-lo2(ct[0]), -lo2(ct[0])), cm = pack2(hi2(ct[0]), hi2(ct[0]));
#pragma unroll
            for (int k = 0; k < E / 2; ++k) {
              const f32x2 tq = fma2(xq[k], c2, nq), tm = fma2(cmb[k], c2, nm);
              const float q0 = ex2_approx(lo2(tq)), q1 = ex2_approx(hi2(tq)), m0 = ex2_approx(lo2(tm)), m1 = ex2_approx(hi2(tm));
              const f32x2 eq = pack2(q0, q1), em = pack2(m0, m1);
              zq = add2(zq, eq);
              zm = add2(zm, em);
              const f32x2 pq = mul2(cq, eq), pm = mul2(cm, em);
              if (lo2(pm) > lo2(pq)) {
                aq += q0;
                am += m0;
              }
              if (hi2(pm) > hi2(pq)) {
                aq += q1;
                am += m1;
              }
            }
            vz[0] = in ? pack2(lo2(zq) + hi2(zq), lo2(zm) + hi2(zm)) : pack2(0.f, 0.f);
            va[0] = in ? pack2(aq, am) : pack2(0.f, 0.f);
          }
          // no term is negative, so a vector that holds a big entry has a big sum
          bool big = false;
#pragma unroll
          for (int q = 0; q < NP; ++q) big = big || lo2(vz[q]) > bt[2 * q] || hi2(vz[q]) > bt[2 * q + 1];
          const int v = (s + t) * 32 + lane;
          const bool ragged = s + t < ce && (v < whole.lo || v >= whole.hi) && v * E < p.V;
          if (big || ragged) {
            if (kLater) {
              later |= 1u << (s + t - c);
              continue;
            }
            slow_vector<DT, ENS, NCH, AL, FORM>(p, kc, u, r[t], v, ragged, !slow, acc);
            slow = true;
          } else {
#pragma unroll
            for (int q = 0; q < NP; ++q) {
              zc[q] = add2(zc[q], vz[q]);
              ac[q] = add2(ac[q], va[q]);
            }
          }
        }
      }
      if constexpr (kShared) {
        if (__any_sync(0xffffffffu, later != 0u)) {
          const int T = blockDim.x;
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            acc[(2 * q) * T] = static_cast<double>(lo2(zc[q])) + (slow ? acc[(2 * q) * T] : 0.0);
            acc[(2 * q + 1) * T] = static_cast<double>(hi2(zc[q])) + (slow ? acc[(2 * q + 1) * T] : 0.0);
            acc[(NCH + 2 * q) * T] = static_cast<double>(lo2(ac[q])) + (slow ? acc[(NCH + 2 * q) * T] : 0.0);
            acc[(NCH + 2 * q + 1) * T] = static_cast<double>(hi2(ac[q])) + (slow ? acc[(NCH + 2 * q + 1) * T] : 0.0);
            zc[q] = ac[q] = pack2(0.f, 0.f);
          }
          slow = true;
          slow_entries<DT, NCH>(kc, u, c, later, acc);
        }
      } else if (kLater) {
#pragma unroll 1
        for (; later; later &= later - 1) {
          Vectors<NR> none;
#pragma unroll
          for (int i = 0; i < NR; ++i) none.r[i] = neg_inf_vector<DT>();
          slow_vector<DT, ENS, NCH, AL, FORM>(p, kc, u, none, (c + __ffs(later) - 1) * 32 + lane, true, !slow, acc);
          slow = true;
        }
      }
      if (ce < end) {  // (the lane's slots take over)
        const int T = blockDim.x;
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          acc[(2 * q) * T] = static_cast<double>(lo2(zc[q])) + (slow ? acc[(2 * q) * T] : 0.0);
          acc[(2 * q + 1) * T] = static_cast<double>(hi2(zc[q])) + (slow ? acc[(2 * q + 1) * T] : 0.0);
          acc[(NCH + 2 * q) * T] = static_cast<double>(lo2(ac[q])) + (slow ? acc[(NCH + 2 * q) * T] : 0.0);
          acc[(NCH + 2 * q + 1) * T] = static_cast<double>(hi2(ac[q])) + (slow ? acc[(NCH + 2 * q + 1) * T] : 0.0);
          zc[q] = ac[q] = pack2(0.f, 0.f);
        }
        slow = true;
      }
    }
    double sums[2 * NCH];
    {
      const int T = blockDim.x;
#pragma unroll
      for (int q = 0; q < NP; ++q) {
        sums[2 * q] = static_cast<double>(lo2(zc[q]));
        sums[2 * q + 1] = static_cast<double>(hi2(zc[q]));
        sums[NCH + 2 * q] = static_cast<double>(lo2(ac[q]));
        sums[NCH + 2 * q + 1] = static_cast<double>(hi2(ac[q]));
      }
      if (slow) {
#pragma unroll
        for (int q = 0; q < 2 * NCH; ++q) sums[q] += acc[q * T];
      }
    }
    __syncwarp();
    const double mine = warp_sums<2 * NCH>(sums, lane);
    if (lane >= 16 && lane % (16 / NCH) == 0) store_cluster(recs + (record_at(rec) * NCH + (lane - 16) / (16 / NCH)) * 8, mine);
    all += mine;
  }
  if (lane < 16 && lane % (16 / NCH) == 0) store_cluster(part + lane / (16 / NCH) * 8, all);
}

// Shared memory of a block, in front of every thread's 2 NCH slots of the slow path.
template <int NCH, int PARTS = kMaxParts, int SUMS = kMaxSums>
struct DrawShared {
  DrawConst kc;
  DrawUnit<NCH> unit;
  // (of the cluster's first block)
  double recs[SUMS / 8 * 9];                 // sums of the chunks (see record_at)
  double part[PARTS * kMaxDrawWarps][NCH];   // shares of the normalisers, of every warp
  double step_mass[32];
  double inv[NCH];      // one over the normalisers
  double base, target;  // mass before the winning chunk; the running total to be reached
  float cf[NCH];        // k / Z
  int win;              // the winning chunk; -1: nothing to draw, -2: no mass, -3: the set of tokens is to be decided again
};

// The share of warp w of W; chunks without steps get sums of zero.  FORM: logit level: bit 0: two models, bit 1: with a mask.
template <int DT, bool ENS, int NCH, bool AL, int FORM, typename SH>
__device__ __forceinline__ void draw_sweep(const KParams& p, SH& sh, int w, int W, double* acc) {
  const int s_lo = static_cast<int>(static_cast<long long>(p.nsteps) * w / W);
  const int s_hi = static_cast<int>(static_cast<long long>(p.nsteps) * (w + 1) / W);
  const unsigned recs = at_first(sh.recs), part = at_first(sh.part[w]);
  const int cs = p.draw_cs, rec = w * p.draw_chunks, used = (s_hi - s_lo + cs - 1) / cs;
  for (int k = used * NCH + (threadIdx.x & 31); k < p.draw_chunks * NCH; k += 32) store_cluster(recs + (record_at(rec + k / NCH) * NCH + k % NCH) * 8, 0.0);
  draw_sweep_as<DT, ENS, NCH, AL, FORM>(p, sh.kc, sh.unit, cs, s_lo, s_hi, acc, rec, recs, part);
}

// The masses of one lane's tokens of step s under the refined normalisers (coefficients cf = k / Z): small ones in fp32; the bits of big
// ones, which are for fp64 (big_mass), with 0 in their place; and the bits of those inside the mask.
template <int DT, bool ENS, int NCH, bool AL, int FORM>
__device__ __forceinline__ void step_masses(const KParams& p, const DrawConst& kc, const DrawUnit<NCH>& u, const float* cf, int s,
                                            Vectors<ENS ? NCH : 2>& rv, float (&m)[Elem<DT>::E], unsigned& bigbits, unsigned& inbits) {
  constexpr int E = Elem<DT>::E, NR = ENS ? NCH : 2;
  const int v = s * 32 + (threadIdx.x & 31);
  const VecRange whole = whole_vectors<DT, AL>(kc.V);
  const bool in = v >= whole.lo && v < whole.hi;
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    rv.r[i] = neg_inf_vector<DT>();
    if (in && i < kc.n) rv.r[i] = load_whole<DT, AL>(u.base + i * kc.row_step, v);
  }
  if (!in && v * E < kc.V) {
#pragma unroll
    for (int i = 0; i < NR; ++i)
      if (i < kc.n) rv.r[i] = load_vector<DT, AL>(u.base + i * kc.row_step, v, kc.V, whole);
  }
  float x[NCH][E];
  vector_args<DT, ENS, NCH, AL, FORM>(p, kc, u, rv, v, x);
  bigbits = inbits = 0u;
#pragma unroll
  for (int k = 0; k < E; ++k) {
    float tot = 0.f;
    bool big = false;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const float e = ex2_approx(fmaf(x[i][k], kc.cT, u.nref[i]));
      big = big || e > u.bt[i];
      tot = __fadd_rn(tot, __fmul_rn(cf[i], e));
    }
    m[k] = big ? 0.f : fmaxf(0.f, tot);
    if (big) bigbits |= 1u << k;
    if (ENS || x[1][k] != -INFINITY) inbits |= 1u << k;
  }
}

// The whole position again by the cluster's first block, for another law or other coefficients.  Rare; out of line.
template <int DT, bool ENS, int NCH, bool AL, int FORM, typename SH>
__device__ __noinline__ void draw_sweep_again(const KParams& p, SH& sh, int W, double* acc) {
  for (int w = threadIdx.x >> 5; w < W; w += blockDim.x >> 5) draw_sweep<DT, ENS, NCH, AL, FORM>(p, sh, w, W, acc);
}

// The normalisers from the shares of all W warps, and the chunk that holds the token.  One warp.  `first_pass`: the set of tokens with a
// positive mass was decided with the streaming launch's normalisers.  A token whose sign that got wrong counts for no more than their
// error (1e-7, a few 1e-6 at low temperature), which matters only where the whole residual mass is below a thousand times that: there
// the set is decided again with the refined ones (sh.win = -3).  (Where the normalisers of all channels are the same number, r is q and
// nothing is left.)
template <bool ENS, int NCH, typename SH>
__device__ __forceinline__ void find_chunk(const KParams& p, SH& sh, int W, bool first_pass) {
  constexpr int G = 32 / NCH;  // lanes of a channel
  const int lane = threadIdx.x & 31, i = lane / G, live = ENS ? p.n : 2;
  const DrawUnit<NCH>& u = sh.unit;
  double z = 0.0;
#pragma unroll 4
  for (int w = lane % G; w < W; w += G) z += sh.part[w][i];
#pragma unroll
  for (int d = G / 2; d > 0; d >>= 1) z += __shfl_xor_sync(0xffffffffu, z, d);
  const double inv = i < live ? 1.0 / z : 0.0, k = i < live ? coefficient<ENS>(p, i, u.pis, u.law) * inv : 0.0;
  if (lane % G == 0) {
    sh.inv[i] = inv;
    sh.cf[i] = static_cast<float>(k);
  }
  double c64[NCH];
#pragma unroll
  for (int q = 0; q < NCH; ++q) c64[q] = __shfl_sync(0xffffffffu, k, q * G);
  auto mass_of = [&](int c) -> double {  // (products rounded one by one: equal sums under opposite coefficients cancel)
    const double* a = &sh.recs[record_at(c) * NCH];
    double m = __dmul_rn(c64[0], a[0]);
#pragma unroll
    for (int q = 1; q < NCH; ++q) m = __dadd_rn(m, __dmul_rn(c64[q], a[q]));
    return m > 0.0 ? m : 0.0;
  };
  // consecutive chunks to a lane; then the chunks of the lane that holds the target, one to a lane (32 and more of them: in a few goes)
  const int chunks = W * p.draw_chunks, per = (chunks + 31) / 32;
  const int c_lo = lane * per, c_hi = c_lo + per < chunks ? c_lo + per : chunks;
  double mine = 0.0;
#pragma unroll 4
  for (int c = c_lo; c < c_hi; ++c) mine += mass_of(c);
  const double incl = running_total<32>(mine, lane);
  const double S = __shfl_sync(0xffffffffu, incl, 31), target = word_to_uniform(u.word) * S;
  // the first that reaches the target; where rounding leaves none, the last with mass
  const unsigned some = __ballot_sync(0xffffffffu, mine > 0.0), hit = __ballot_sync(0xffffffffu, mine > 0.0 && incl >= target);
  const int who = hit ? __ffs(hit) - 1 : 31 - __clz(some);
  double base = __shfl_sync(0xffffffffu, incl - mine, who & 31), win_base = 0.0;
  int win = -1;
  const int w_lo = (who & 31) * per, w_hi = w_lo + per < chunks ? w_lo + per : chunks;
#pragma unroll 1
  for (int c0 = w_lo; c0 < w_hi && some != 0u; c0 += 32) {
    const double m = c0 + lane < w_hi ? mass_of(c0 + lane) : 0.0, in = running_total<32>(m, lane);
    const unsigned with = __ballot_sync(0xffffffffu, m > 0.0), ok = __ballot_sync(0xffffffffu, m > 0.0 && base + in >= target);
    if (with) {
      const int k = ok ? __ffs(ok) - 1 : 31 - __clz(with);
      win = c0 + k;
      win_base = base + __shfl_sync(0xffffffffu, in - m, k);
    }
    if (ok) break;
    base += __shfl_sync(0xffffffffu, in, 31);
  }
  bool again = false;
  if (first_pass && u.law == kDrawResidual) {  // (the whole warp)
    const bool off = i < live && fabs(z * kBigShare - static_cast<double>(u.bt[i])) * 1000.0 > S * static_cast<double>(u.bt[i]);
    const double z0 = __shfl_sync(0xffffffffu, z, 0);
    const unsigned offs = __ballot_sync(0xffffffffu, off), unlike = __ballot_sync(0xffffffffu, i < live && z != z0);
    again = offs != 0u && unlike != 0u;
  }
  if (lane == 0) {
    sh.win = some != 0u && S > 0.0 ? win : -2;
    sh.base = win_base;
    sh.target = target;
    if (!u.emit) sh.win = -1;
    if (again) sh.win = -3;
    if (p.diag && u.j != p.gamma && u.law == kDrawResidual) p.diag[static_cast<long long>(u.uidx) * 4 + 3] = static_cast<float>(S);
  }
}

// The rest of a position, after the sweep: the block that has the sums finds the chunk, the step and the token.
template <int DT, bool ENS, int NCH, bool AL, int FORM, typename SH>
__device__ __forceinline__ void locate(const KParams& p, SH& sh, double* acc) {
  constexpr int E = Elem<DT>::E;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int W = p.draw_parts * nw;
  DrawUnit<NCH>& u = sh.unit;
  const int cs = p.draw_cs;
#pragma unroll 1
  for (int pass = 0; pass < 3; ++pass) {
    if (warp == 0) find_chunk<ENS, NCH>(p, sh, W, pass == 0);
    __syncthreads();
    const int win = sh.win;
    if (win == -1) return;
    if (win < 0) {
      // no residual mass although a token is needed: this block draws from r instead, over the whole position
      if (u.law != kDrawResidual) return;
      __syncthreads();
      if (tid == 0 && win == -3) {
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
          u.ct[i] = sh.cf[i];
          u.ck[i] = coefficient<ENS>(p, i, u.pis, kDrawResidual) * sh.inv[i];
        }
      } else if (tid == 0) {
        // (this thread alone, after it or an earlier launch wrote the row's status, which may lie in host memory: no atomic)
        if (!u.accepted) p.row_status[u.b] |= static_cast<unsigned>(COS_ROW_RESIDUAL_EMPTY);
        u.law = kDrawR;
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
          u.ck[i] = coefficient<ENS>(p, i, u.pis, kDrawR) * sh.inv[i];
          u.ct[i] = static_cast<float>(u.ck[i]);
        }
      }
      __syncthreads();
      draw_sweep_again<DT, ENS, NCH, AL, FORM>(p, sh, W, acc);
      __syncthreads();
      continue;
    }
    const double* inv = sh.inv;
    const float* cf = sh.cf;
    const double target = sh.target;
    // the steps of that chunk, dealt out over the warps in up to 32 records of `gsz` steps (one step, nearly always)
    const int ww = win / p.draw_chunks;
    const int s0 = static_cast<int>(static_cast<long long>(p.nsteps) * ww / W) + win % p.draw_chunks * cs;
    const int end = static_cast<int>(static_cast<long long>(p.nsteps) * (ww + 1) / W);
    const int s1 = s0 + cs < end ? s0 + cs : end, gsz = (cs + 31) / 32;
    // the first lane whose total `in` (its own mass: m) reaches the target, or the last with mass where rounding leaves none
    auto first_reach = [&](double m, double in, double from, double& upto) -> int {
      const unsigned some = __ballot_sync(0xffffffffu, m > 0.0), ok = __ballot_sync(0xffffffffu, m > 0.0 && from + in >= target);
      const int k = ok ? __ffs(ok) - 1 : 31 - __clz(some);
      upto = from + __shfl_sync(0xffffffffu, in - m, k & 31);
      return ok ? k : k - 32;  // (negative: not reached; -33: no mass at all)
    };
    // (what the lanes of this warp hold of step `held`: their masses, the running total, the masses of their tokens)
    double own = 0.0, in = 0.0;
    int held = -1;
    Vectors<ENS ? NCH : 2> rv;
    float m[E];
    unsigned bigbits = 0u, inbits = 0u;
    auto hold = [&](int s) {
      step_masses<DT, ENS, NCH, AL, FORM>(p, sh.kc, u, cf, s, rv, m, bigbits, inbits);
      own = 0.0;
#pragma unroll
      for (int k = 0; k < E; ++k) own += static_cast<double>(m[k]);
#pragma unroll 1
      for (unsigned bits = bigbits; bits; bits &= bits - 1) {
        const int k = __ffs(bits) - 1;
        own += big_mass<DT, ENS, NCH, FORM>(sh.kc, u, inv, rv, (s * 32 + lane) * E + k, k, (inbits >> k) & 1u);
      }
      in = running_total<32>(own, lane);
      held = s;
    };
#pragma unroll 1
    for (int t = warp; s0 + t * gsz < s1; t += nw) {
      double rm = 0.0;
#pragma unroll 1
      for (int s = s0 + t * gsz; s < s0 + (t + 1) * gsz && s < s1; ++s) {
        hold(s);
        rm += __shfl_sync(0xffffffffu, in, 31);
      }
      if (lane == 0) sh.step_mass[t] = rm;
    }
    __syncthreads();
    if (held < 0) return;  // (no step of the chunk is this warp's)
    double at;
    const double sm = (s0 + lane * gsz < s1) ? sh.step_mass[lane] : 0.0;
    const int k = first_reach(sm, running_total<32>(sm, lane), sh.base, at);
    if (k == -33) return;
    if ((k & 31) % nw != warp) return;
    // one warp goes on: the record's steps in order, the lanes of a step, the tokens of a lane's vector
    const int g0 = s0 + (k & 31) * gsz, g1 = g0 + gsz < s1 ? g0 + gsz : s1;
    int some = -1;  // the last step with mass, and the total before it
    double some_at = 0.0;
#pragma unroll 1
    for (int s = g0;;) {
      if (s != held) hold(s);
      double before;
      const int l = first_reach(own, in, at, before);
      if (l != -33) {
        some = s;
        some_at = at;
      }
      if (l < 0) {  // (not reached in this step)
        at += __shfl_sync(0xffffffffu, in, 31);
        if (++s < g1) continue;
        if (some < 0) return;
        if (some != held) hold(some);  // (rounding left none that reaches the target: the last token with mass)
        first_reach(own, in, some_at, before);
      }
      const unsigned with = __ballot_sync(0xffffffffu, own > 0.0);
      const int who = l >= 0 ? l : 31 - __clz(with);
      if (lane == who) {
        double run = before;
        int last = -1;
        bool reached = false;
        auto take = [&](int q, double mass) {
          run += mass;
          if (mass > 0.0 && !reached) {
            last = q;
            reached = run >= target;
          }
        };
        const int e0 = (held * 32 + lane) * E;
        if (bigbits == 0u) {
#pragma unroll
          for (int q = 0; q < E; ++q) take(q, static_cast<double>(m[q]));
        } else {
#pragma unroll 1
          for (int q = 0; q < E; ++q) {
            float small = m[0];
#pragma unroll
            for (int r = 1; r < E; ++r) small = r == q ? m[r] : small;
            take(q, (bigbits >> q) & 1u ? big_mass<DT, ENS, NCH, FORM>(sh.kc, u, inv, rv, e0 + q, q, (inbits >> q) & 1u) : static_cast<double>(small));
          }
        }
        if (last >= 0) {
          p.out_tokens[u.uidx] = e0 + last;
          // Algorithm 2's Score returns the bonus token with its probability under the law it came from
          if (u.j == p.gamma && p.bonus_prob != nullptr)
            p.bonus_prob[u.b] = static_cast<float>(big_mass<DT, ENS, NCH, FORM>(sh.kc, u, inv, rv, e0 + last, last, (inbits >> last) & 1u));
        }
      }
      return;
    }
  }
}

// The block's position from the records of the streaming launch (and the row's outputs, see decide_row): every block decides
// its row for itself.  False when there is nothing to draw.
template <int DT, bool ENS, int NCH, typename SH, typename R>
__device__ __forceinline__ bool decide_unit_to_draw(const KParams& p, SH& sh, RowShared& rs, const TilePlan& t, const TileInputs& in, int b, int want,
                                                    int part, R ready) {
  const int tid = threadIdx.x;
  DrawUnit<NCH>& u = sh.unit;
  decide_sampled<DT, ENS ? kEnsembleSample : kLogitSample, 4>(
      p, rs, t, in, b, want, ready,
      [&](const PairStats* f, int j, int pi, unsigned word, int accepted, int drawable) {
        const int pis = (pi >= 0 && pi < p.n) ? pi : 0;
        const int law = (j == p.gamma) ? (p.bonus_model >= 0 ? kDrawQ : kDrawR) : kDrawResidual;
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
          const bool live = i < (ENS ? p.n : 2);
          const double ck = live ? coefficient<ENS>(p, i, pis, law) * f[i].inv : 0.0;
          u.nref[i] = live ? -f[i].ref : 0.f;
          u.bt[i] = live ? static_cast<float>(f[i].s * kBigShare) : INFINITY;
          u.ck[i] = ck;
          u.ct[i] = static_cast<float>(ck);
        }
        u.b = b;
        u.j = j;
        u.uidx = b * p.P + j;
        u.pis = pis;
        u.law = law;
        u.word = word;
        u.accepted = accepted;
        u.drawable = drawable;
        u.thr = (!ENS && p.mask_model >= 0) ? f[1].thr : -INFINITY;
        u.base = reinterpret_cast<const char*>(p.logits) +
                 (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
      },
      [&](int a) { return part == 0 && (want < 0 || want == a); }, [&](int j) { return part == 0 && (want < 0 || want == j); });
  const bool emit = (rs.a == u.j);
  if (tid == 0) u.emit = emit ? 1 : 0;
  return u.drawable && (emit || u.j != p.gamma);
}

// One cluster of p.draw_parts blocks for each position.  All blocks of a cluster take the same way, and so meet at its barriers.
template <int DT, bool ENS, int NCH, bool AL, int FORM>
__global__ void __launch_bounds__(NCH == 8 ? 256 : kMaxDrawThreads, NCH == 2 ? 2 : (NCH == 4 ? 1 : 2)) cos_draw_kernel(const __grid_constant__ KParams p) {
  extern __shared__ __align__(16) unsigned char draw_smem_raw[];
  DrawShared<NCH>& sh = *reinterpret_cast<DrawShared<NCH>*>(draw_smem_raw);
  double* slots = reinterpret_cast<double*>(draw_smem_raw + sizeof(DrawShared<NCH>));
  double* acc = slots + threadIdx.x;
  const int slot = blockIdx.x / p.draw_parts, rank = blockIdx.x % p.draw_parts, nw = blockDim.x >> 5;
  fill_const<DT>(p, sh.kc);
  cluster_arrive();  // (the first block has begun: its shared memory may be written to)
  // launched while the kernel before it drains; nothing but inputs is read before that one is complete
  bool draws;
  if (NCH != 8 && p.decide) {
    RowShared& rs = *reinterpret_cast<RowShared*>(slots);
    int b = slot, want = -1;
    if (p.draw_all) {
      const int drafts = p.B * p.gamma;  // every draft position, then the bonus positions
      b = slot < drafts ? slot / p.gamma : slot - drafts;
      want = slot < drafts ? slot % p.gamma : p.gamma;
    }
    constexpr int kMode = ENS ? kEnsembleSample : kLogitSample;
    const TilePlan t = tile_plan<kMode>(p);
    draws = decide_unit_to_draw<DT, ENS, NCH>(p, sh, rs, t, tile_inputs<DT, kMode>(p, t, b, 0), b, want, rank,
                                              [] { asm volatile("griddepcontrol.wait;" ::: "memory"); });
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    DrawUnit<NCH> d;
    draws = load_unit<DT, ENS, NCH>(p, slot, d);
    if (threadIdx.x == 0) sh.unit = d;
  }
  cluster_wait();
  if (!draws) return;
  __syncthreads();
  draw_sweep<DT, ENS, NCH, AL, FORM>(p, sh, rank * nw + (threadIdx.x >> 5), p.draw_parts * nw, acc);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cluster_arrive();
  cluster_wait();
  if (rank == 0) {
    __syncthreads();
    locate<DT, ENS, NCH, AL, FORM>(p, sh, acc);
  }
}

// Test hook: the combined distribution of every position, token by token, from the statistics the streaming launch left.
template <int DT>
__global__ void __launch_bounds__(256) cos_dump_kernel(const __grid_constant__ KParams p, bool ens) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int uidx = blockIdx.y, b = uidx / p.P, j = uidx % p.P;
  const UnitStats* st = &p.ustats[uidx];
  if (!p.unit_res[uidx].w) return;
  const char* base = reinterpret_cast<const char*>(p.logits) +
                     (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
  float* out = p.dump_r + static_cast<long long>(uidx) * p.V;
  const long long row_step = p.s_model * Elem<DT>::bytes;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < p.V; x += gridDim.x * blockDim.x) {
    float r = 0.f;
    if (ens) {
      for (int i = 0; i < p.n; ++i)
        r = fmaf(static_cast<float>(p.w64[i] / st->s[i]), ex2_approx(fmaf(Elem<DT>::load1(base + i * row_step, x), p.cT, -st->ref[i])), r);
    } else {
      float cmb = 0.f;
      bool in = true;
      for (int i = 0; i < p.n; ++i) {
        const float l = Elem<DT>::load1(base + i * row_step, x);
        cmb = fmaf(p.w[i], l, cmb);
        if (i == p.mask_model) in = l >= st->thr32;
      }
      r = in ? ex2_approx(fmaf(cmb, p.cT, -st->ref[1])) * static_cast<float>(1.0 / st->s[1]) : 0.f;
    }
    out[x] = r;
  }
}

}  // namespace cosv

#endif  // COS_DRAW_CUH
