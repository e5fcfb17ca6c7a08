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
// The part behind the sweep is a chain of latencies, issue slots and instruction fetches (counted on one row of 151936 tokens: most
// stalls are for instructions), so what can be done by one warp is, and nothing is unrolled that need not be.
// Measured (64 rows of 2 x 151936 tokens): 9 us of sweep, 3 until the cluster's last warp is done, 6 to find the token.  Records in
// global memory and the last block to report (fence and counter) took 5 us longer; two more barriers of the cluster, for all
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

// What the functions that are not inlined need of the parameters, in shared memory: behind a call the parameters are no longer
// operands from the constant bank but loads through a generic address, a trip to L2 for each line of them the first time.
struct DrawConst {
  long long row_step;  // bytes from one model's row to the next
  double cT64, w64[COS_MAX_MODELS];
  float cT, w[COS_MAX_MODELS];
  int n, V, mask_model;
};

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

// The arguments of the channels for one token.
template <int DT, bool ENS, int NCH>
__device__ __forceinline__ void entry_args(const DrawConst& p, const DrawUnit<NCH>& u, int e, float (&x)[NCH]) {
  if (ENS) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      x[i] = -INFINITY;
      if (i < p.n) x[i] = Elem<DT>::load1(u.base + i * p.row_step, e);
    }
  } else {
    const float l0 = Elem<DT>::load1(u.base, e);
    float l1 = 0.f, gate = l0;
    if (p.n >= 2) l1 = Elem<DT>::load1(u.base + p.row_step, e);
    x[0] = u.pis == 0 ? l0 : l1;
    if (p.mask_model == 1) gate = l1;
    x[1] = __fmul_rn(p.w[0], l0);
    if (p.n >= 2) x[1] = fmaf(p.w[1], l1, x[1]);
    for (int i = 2; i < p.n; ++i) {
      const float l = Elem<DT>::load1(u.base + i * p.row_step, e);
      if (i == u.pis) x[0] = l;
      if (i == p.mask_model) gate = l;
      x[1] = fmaf(p.w[i], l, x[1]);
    }
    if (p.mask_model >= 0 && !(gate >= u.thr)) x[1] = -INFINITY;
  }
}

// fp64 terms of one token (its arguments: x): e_i of every channel.  For "big" tokens (more than 2^-8 of a normaliser) and the
// bonus token's probability.
template <int DT, bool ENS, int NCH>
__device__ __forceinline__ void exact_terms(const DrawConst& p, const DrawUnit<NCH>& u, int e, const float (&x)[NCH], double (&out)[NCH]) {
  double t[NCH];
#pragma unroll
  for (int i = 0; i < NCH; ++i) t[i] = static_cast<double>(x[i]);
  if (!ENS && !(x[1] == -INFINITY)) {  // (the combination again, in fp64)
    t[1] = 0.0;
    for (int i = 0; i < p.n; ++i) t[1] = fma(p.w64[i], static_cast<double>(Elem<DT>::load1(u.base + i * p.row_step, e)), t[1]);
  }
#pragma unroll 1
  for (int k = 0; k < NCH; ++k) {  // (one copy of the exponential)
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < NCH; ++i)
      if (i == k) v = t[i] * p.cT64 + static_cast<double>(u.nref[i]);
    v = exp2(v);
#pragma unroll
    for (int i = 0; i < NCH; ++i)
      if (i == k) out[i] = v;
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

// The arguments of the NCH channels for the E tokens of vector v (any vector of the row; -inf beyond V), one lane.
template <int DT, bool ENS, int NCH, bool AL>
__device__ __forceinline__ void vector_args(const KParams& p, const DrawUnit<NCH>& u, int v, float (&x)[NCH][Elem<DT>::E]) {
  constexpr int E = Elem<DT>::E;
  const VecRange whole = whole_vectors<DT, AL>(p.V);
  const long long row_step = p.s_model * Elem<DT>::bytes;
  if (ENS) {
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      uint4 r = neg_inf_vector<DT>();
      if (i < p.n) r = load_vector<DT, AL>(u.base + i * row_step, v, p.V, whole);
#pragma unroll
      for (int k = 0; k < E; ++k) x[i][k] = entry<DT>(r, k);
    }
  } else {
    auto row = [&](int i) { return load_vector<DT, AL>(u.base + i * row_step, v, p.V, whole); };
    const uint4 r0 = row(0);
    const uint4 r1 = p.n >= 2 ? row(1) : r0;
    f32x2 xq[E / 2], cmb[E / 2];
    const LogitWeights lw = logit_weights(p, u.pis, u.thr);
    if (p.mask_model >= 0)
      logit_args<DT, false, true>(p, lw, r0, r1, row, xq, cmb);
    else
      logit_args<DT, false, false>(p, lw, r0, r1, row, xq, cmb);
#pragma unroll
    for (int k = 0; k < E; ++k) {  // (beyond V the combination of -inf could be anything)
      x[0][k] = pair_at(xq[k / 2], k);
      x[1][k] = (v * E + k < p.V) ? pair_at(cmb[k / 2], k) : -INFINITY;
    }
  }
}

// The mass of one big token.  Out of line.
template <int DT, bool ENS, int NCH>
__device__ __noinline__ double big_mass(const DrawConst& p, const DrawUnit<NCH>& u, const double* inv, int e) {
  float x[NCH];
  double d[NCH];
  entry_args<DT, ENS, NCH>(p, u, e, x);
  exact_terms<DT, ENS, NCH>(p, u, e, x, d);
  return exact_mass<ENS, NCH>(p, d, inv, u.pis, u.law);
}

// The vectors the fast loop left out (bit k of a lane's `slow`: its vector of step c + k): those with a big entry, which is summed in
// fp64 then, and the ragged ends of the row.  The warp takes 32 entries at a time, one a lane; the sums go to the lanes'
// slots of `acc`.  Out of line.  (One lane going through its vector while the others waited took 2 us a vector, and the warp that
// happened on most big tokens was the last of its cluster by 5 to 8 us.)
template <int DT, bool ENS, int NCH>
__device__ __noinline__ void slow_vectors(const DrawConst& p, const DrawUnit<NCH>& u, int c, unsigned slow, double* acc) {
  constexpr int E = Elem<DT>::E, G = 32 / E;
  const int T = blockDim.x, lane = threadIdx.x & 31;
  for (unsigned any = __reduce_or_sync(0xffffffffu, slow); any; any &= any - 1) {
    const int k = __ffs(any) - 1;
    unsigned m = __ballot_sync(0xffffffffu, (slow >> k) & 1u);
    while (m) {
      unsigned t = m;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        if (q < lane / E) t &= t - 1;
        m &= m - 1;
      }
      const int e = t ? ((c + k) * 32 + __ffs(t) - 1) * E + lane % E : p.V;
      if (e < p.V) {
        float x[NCH], f[NCH], tot = 0.f;
        bool big = false;
        entry_args<DT, ENS, NCH>(p, u, e, x);
#pragma unroll
        for (int i = 0; i < NCH; ++i) {
          f[i] = ex2_approx(fmaf(x[i], p.cT, u.nref[i]));
          big = big || f[i] > u.bt[i];
          tot = __fadd_rn(tot, __fmul_rn(u.ct[i], f[i]));
        }
        double d[NCH];
#pragma unroll
        for (int i = 0; i < NCH; ++i) d[i] = static_cast<double>(f[i]);
        bool counts = tot > 0.f;
        if (big) {
          exact_terms<DT, ENS, NCH>(p, u, e, x, d);
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
}

// The steps [s_lo, s_hi) of a position by one warp, in chunks of cs steps: per channel the sum over the tokens with a positive mass,
// for every chunk NCH sums to rec, and to part the normaliser's share, of all chunks together (both in the cluster's first block).
// The fast loop adds vectors up in fp32; vectors that need the slow path it only remembers until the end of the strip (their
// sums, in fp64, in the thread's slots of `acc`).
// What bounds it: instruction issue (counted at logit level, 128 rows of 256000 tokens: 211 instructions a step, 0.53 of the issue
// slots of the average multiprocessor, 0.67 of the busiest).  Loads in flight do not: fetching a step as soon as a place is free,
// so that two are always on their way, gained nothing with two channels and lost 2 to 7 % with four.
// PAIR, MASKED: logit level with exactly two models, and with a mask.
template <int DT, bool ENS, int NCH, bool AL, bool PAIR, bool MASKED>
__device__ __forceinline__ void draw_sweep_as(const KParams& p, const DrawConst& kc, const DrawUnit<NCH>& u, int cs, int s_lo, int s_hi, double* acc,
                                              unsigned rec, unsigned part) {
  constexpr int E = Elem<DT>::E;
  constexpr int NP = NCH / 2;
  constexpr int NR = ENS ? NCH : 2;         // vectors of a step kept in registers
  constexpr int US = (NR == 2) ? 2 : 1;     // steps fetched at a time
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
  for (int begin = s_lo; begin < s_hi; begin += cs, rec += NCH * 8) {
    const int end = begin + cs < s_hi ? begin + cs : s_hi;
    double sums[2 * NCH];
    // in strips of 32 steps: a bit each in the slow-path mask
    for (int c = begin; c < end; c += 32) {
      const int ce = c + 32 < end ? c + 32 : end;
      unsigned slow = 0u;
      f32x2 zc[NP], ac[NP];
#pragma unroll
      for (int q = 0; q < NP; ++q) zc[q] = ac[q] = pack2(0.f, 0.f);
      for (int s = c; s < ce; s += US) {
        uint4 r[US][NR];
#pragma unroll
        for (int t = 0; t < US; ++t) {
          const int v = (s + t) * 32 + lane;
          const bool in = v >= whole.lo && v < whole.hi;
#pragma unroll
          for (int i = 0; i < NR; ++i) {
            r[t][i] = neg_inf_vector<DT>();
            if (in && s + t < ce && i < p.n) r[t][i] = load_whole<DT, AL>(base + i * row_step, v);
          }
          if (!in && s + t < ce) slow |= 1u << (s + t - c);
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
                const f32x2 arg = fma2(pack2(entry<DT>(r[t][2 * q], k), entry<DT>(r[t][2 * q + 1], k)), c2, nref[q]);
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
            logit_args<DT, PAIR, MASKED>(p, lw, r[t][0], r[t][1],
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
          if (big) {
            slow |= 1u << (s + t - c);
          } else {
#pragma unroll
            for (int q = 0; q < NP; ++q) {
              zc[q] = add2(zc[q], vz[q]);
              ac[q] = add2(ac[q], va[q]);
            }
          }
        }
      }
      const int T = blockDim.x;
      const bool more = c > begin;
#pragma unroll
      for (int q = 0; q < NP; ++q) {
        sums[2 * q] = static_cast<double>(lo2(zc[q])) + (more ? acc[(2 * q) * T] : 0.0);
        sums[2 * q + 1] = static_cast<double>(hi2(zc[q])) + (more ? acc[(2 * q + 1) * T] : 0.0);
        sums[NCH + 2 * q] = static_cast<double>(lo2(ac[q])) + (more ? acc[(NCH + 2 * q) * T] : 0.0);
        sums[NCH + 2 * q + 1] = static_cast<double>(hi2(ac[q])) + (more ? acc[(NCH + 2 * q + 1) * T] : 0.0);
      }
      if (ce < end || __any_sync(0xffffffffu, slow != 0u)) {
#pragma unroll
        for (int q = 0; q < 2 * NCH; ++q) acc[q * T] = sums[q];
        slow_vectors<DT, ENS, NCH>(kc, u, c, slow, acc);
#pragma unroll
        for (int q = 0; q < 2 * NCH; ++q) sums[q] = acc[q * T];
      }
    }
    __syncwarp();
    const double mine = warp_sums<2 * NCH>(sums, lane);
    if (lane >= 16 && lane % (16 / NCH) == 0) store_cluster(rec + (lane - 16) / (16 / NCH) * 8, mine);
    all += mine;
  }
  if (lane < 16 && lane % (16 / NCH) == 0) store_cluster(part + lane / (16 / NCH) * 8, all);
}

// Shared memory of a block, in front of every thread's 2 NCH slots of the slow path.
template <int NCH>
struct DrawShared {
  DrawConst kc;
  DrawUnit<NCH> unit;
  // (of the cluster's first block)
  double recs[kMaxSums];                         // sums of the chunks
  double part[kMaxParts * kMaxDrawWarps][NCH];   // shares of the normalisers, of every warp
  double step_mass[32];
  double inv[NCH];      // one over the normalisers
  double base, target;  // mass before the winning chunk; the running total to be reached
  float cf[NCH];        // k / Z
  int win;              // the winning chunk; -1: nothing to draw, -2: no mass, -3: the set of tokens is to be decided again
};

// The share of warp w of W; chunks without steps get sums of zero.
template <int DT, bool ENS, int NCH, bool AL>
__device__ __forceinline__ void draw_sweep(const KParams& p, DrawShared<NCH>& sh, int w, int W, double* acc) {
  const int s_lo = static_cast<int>(static_cast<long long>(p.nsteps) * w / W);
  const int s_hi = static_cast<int>(static_cast<long long>(p.nsteps) * (w + 1) / W);
  const unsigned rec = at_first(&sh.recs[w * p.draw_chunks * NCH]), part = at_first(sh.part[w]);
  const int cs = p.draw_cs, used = (s_hi - s_lo + cs - 1) / cs;
  for (int k = used * NCH + (threadIdx.x & 31); k < p.draw_chunks * NCH; k += 32) store_cluster(rec + k * 8, 0.0);
  const DrawUnit<NCH>& u = sh.unit;
  if (ENS) return draw_sweep_as<DT, ENS, NCH, AL, true, false>(p, sh.kc, u, cs, s_lo, s_hi, acc, rec, part);
  if (p.n == 2 && p.mask_model < 0) return draw_sweep_as<DT, ENS, NCH, AL, true, false>(p, sh.kc, u, cs, s_lo, s_hi, acc, rec, part);
  if (p.n == 2) return draw_sweep_as<DT, ENS, NCH, AL, true, true>(p, sh.kc, u, cs, s_lo, s_hi, acc, rec, part);
  if (p.mask_model < 0) return draw_sweep_as<DT, ENS, NCH, AL, false, false>(p, sh.kc, u, cs, s_lo, s_hi, acc, rec, part);
  draw_sweep_as<DT, ENS, NCH, AL, false, true>(p, sh.kc, u, cs, s_lo, s_hi, acc, rec, part);
}

// The mass of one lane's tokens of step s under the refined normalisers (coefficients cf = k / Z): small ones in fp32, big
// ones in fp64.
template <int DT, bool ENS, int NCH, bool AL>
__device__ __forceinline__ double step_mass(const KParams& p, const DrawConst& kc, const DrawUnit<NCH>& u, const float* cf, const double* inv, int s) {
  constexpr int E = Elem<DT>::E;
  const int v = s * 32 + (threadIdx.x & 31);
  float x[NCH][E];
  vector_args<DT, ENS, NCH, AL>(p, u, v, x);
  unsigned bigbits = 0u;
  float ls = 0.f;
#pragma unroll
  for (int k = 0; k < E; ++k) {
    float tot = 0.f;
    bool big = false;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const float e = ex2_approx(fmaf(x[i][k], p.cT, u.nref[i]));
      big = big || e > u.bt[i];
      tot = __fadd_rn(tot, __fmul_rn(cf[i], e));
    }
    ls += big ? 0.f : fmaxf(0.f, tot);
    bigbits |= big ? (1u << k) : 0u;
  }
  double own = static_cast<double>(ls);
  for (; bigbits; bigbits &= bigbits - 1) own += big_mass<DT, ENS, NCH>(kc, u, inv, v * E + __ffs(bigbits) - 1);
  return own;
}
template <int DT, bool ENS, int NCH>
__device__ __forceinline__ double token_mass(const DrawConst& p, const DrawUnit<NCH>& u, const float* cf, const double* inv, int e) {
  float x[NCH], tot = 0.f;
  bool big = false;
  entry_args<DT, ENS, NCH>(p, u, e, x);
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const float f = ex2_approx(fmaf(x[i], p.cT, u.nref[i]));
    big = big || f > u.bt[i];
    tot = __fadd_rn(tot, __fmul_rn(cf[i], f));
  }
  return big ? big_mass<DT, ENS, NCH>(p, u, inv, e) : static_cast<double>(fmaxf(0.f, tot));
}

// The whole position again by the cluster's first block, for another law or other coefficients.  Rare; out of line.
template <int DT, bool ENS, int NCH, bool AL>
__device__ __noinline__ void draw_sweep_again(const KParams& p, DrawShared<NCH>& sh, int W, double* acc) {
  for (int w = threadIdx.x >> 5; w < W; w += blockDim.x >> 5) draw_sweep<DT, ENS, NCH, AL>(p, sh, w, W, acc);
}

// The normalisers from the shares of all W warps, and the chunk that holds the token.  One warp.  `first_pass`: the set of tokens with a
// positive mass was decided with the streaming launch's normalisers.  A token whose sign that got wrong counts for no more than their
// error (1e-7, a few 1e-6 at low temperature), which matters only where the whole residual mass is below a thousand times that: there
// the set is decided again with the refined ones (sh.win = -3).  (Where the normalisers of all channels are the same number, r is q and
// nothing is left.)
template <bool ENS, int NCH>
__device__ __forceinline__ void find_chunk(const KParams& p, DrawShared<NCH>& sh, int W, bool first_pass) {
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
    const double* a = &sh.recs[c * NCH];
    double m = __dmul_rn(c64[0], a[0]);
#pragma unroll
    for (int q = 1; q < NCH; ++q) m = __dadd_rn(m, __dmul_rn(c64[q], a[q]));
    return fmax(0.0, m);
  };
  // consecutive chunks to a lane, their masses in the place of their first sums
  const int chunks = W * p.draw_chunks, per = (chunks + 31) / 32;
  const int c_lo = lane * per, c_hi = c_lo + per < chunks ? c_lo + per : chunks;
  double mine = 0.0;
#pragma unroll 4
  for (int c = c_lo; c < c_hi; ++c) {
    const double m = mass_of(c);
    sh.recs[c * NCH] = m;
    mine += m;
  }
  double incl = mine;
#pragma unroll 1
  for (int d = 1; d < 32; d <<= 1) {
    const double o = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += o;
  }
  const double S = __shfl_sync(0xffffffffu, incl, 31), target = word_to_uniform(u.word) * S;
  // the first chunk whose running total reaches the target; where rounding leaves none, the last chunk with mass
  double before = incl - mine, base = 0.0;
  int first = -1, last = -1;
  if (mine > 0.0)
#pragma unroll 1
    for (int c = c_lo; c < c_hi; ++c) {
      const double m = sh.recs[c * NCH];
      if (m > 0.0 && first < 0) {
        last = c;
        base = before;
        if (before + m >= target) first = c;
      }
      before += m;
    }
  bool again = false;
  if (first_pass && u.law == kDrawResidual) {  // (the whole warp)
    const bool off = i < live && fabs(z * kBigShare - static_cast<double>(u.bt[i])) * 1000.0 > S * static_cast<double>(u.bt[i]);
    const double z0 = __shfl_sync(0xffffffffu, z, 0);
    const unsigned offs = __ballot_sync(0xffffffffu, off), unlike = __ballot_sync(0xffffffffu, i < live && z != z0);
    again = offs != 0u && unlike != 0u;
  }
  const unsigned hit = __ballot_sync(0xffffffffu, first >= 0), some = __ballot_sync(0xffffffffu, last >= 0);
  const int winner = hit ? __ffs(hit) - 1 : 31 - __clz(some);
  if (some != 0u ? lane == winner : lane == 0) {
    sh.win = some != 0u && S > 0.0 ? last : -2;
    sh.base = base;
    sh.target = target;
    if (!u.emit) sh.win = -1;
    if (again) sh.win = -3;
    if (p.diag && u.j != p.gamma && u.law == kDrawResidual) p.diag[static_cast<long long>(u.uidx) * 4 + 3] = static_cast<float>(S);
  }
}

// The rest of a position, after the sweep: the block that has the sums finds the chunk, the step and the token.
template <int DT, bool ENS, int NCH, bool AL>
__device__ __forceinline__ void locate(const KParams& p, DrawShared<NCH>& sh, double* acc) {
  constexpr int E = Elem<DT>::E;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  const int live = ENS ? p.n : 2, W = p.draw_parts * nw;
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
      draw_sweep_again<DT, ENS, NCH, AL>(p, sh, W, acc);
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
    // running total over the first `lanes` lanes
    auto scan = [&](double m, int lanes) -> double {
#pragma unroll 1
      for (int d = 1; d < lanes; d <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, m, d);
        if (lane >= d) m += o;
      }
      return m;
    };
    // the first lane whose total `in` (its own mass: m) reaches the target, or the last with mass where rounding leaves none
    auto first_reach = [&](double m, double in, double from, double& upto) -> int {
      const unsigned some = __ballot_sync(0xffffffffu, m > 0.0), ok = __ballot_sync(0xffffffffu, m > 0.0 && from + in >= target);
      const int k = ok ? __ffs(ok) - 1 : 31 - __clz(some);
      upto = from + __shfl_sync(0xffffffffu, in - m, k & 31);
      return ok ? k : k - 32;  // (negative: not reached; -33: no mass at all)
    };
    double own = 0.0, in = 0.0;
    int held = -1;  // the step whose masses, and their running total, the lanes of this warp hold
#pragma unroll 1
    for (int t = warp; s0 + t * gsz < s1; t += nw) {
      double rm = 0.0;
#pragma unroll 1
      for (int s = s0 + t * gsz; s < s0 + (t + 1) * gsz && s < s1; ++s) {
        own = step_mass<DT, ENS, NCH, AL>(p, sh.kc, u, cf, inv, s);
        in = scan(own, 32);
        rm += __shfl_sync(0xffffffffu, in, 31);
        held = s;
      }
      if (lane == 0) sh.step_mass[t] = rm;
    }
    __syncthreads();
    if (held < 0) return;  // (no step of the chunk is this warp's)
    double at, m = (s0 + lane * gsz < s1) ? sh.step_mass[lane] : 0.0;
    int k = first_reach(m, scan(m, (s1 - s0 + gsz - 1) / gsz), sh.base, at);
    if (k == -33) return;
    if ((k & 31) % nw != warp) return;
    // one warp goes on: the record's steps in order, the lanes of a step, the tokens of a lane's vector
    const int g0 = s0 + (k & 31) * gsz, g1 = g0 + gsz < s1 ? g0 + gsz : s1;
    int step = -1, who = 0;
    double before = 0.0;
#pragma unroll 1
    for (int s = g0; s < g1; ++s) {
      if (s != held) {
        own = step_mass<DT, ENS, NCH, AL>(p, sh.kc, u, cf, inv, s);
        in = scan(own, 32);
        held = s;
      }
      double upto;
      const int l = first_reach(own, in, at, upto);
      if (l != -33) {
        step = s;
        who = l & 31;
        before = upto;
      }
      if (l >= 0) break;
      at += __shfl_sync(0xffffffffu, in, 31);
    }
    if (step < 0) return;
    const int e = (step * 32 + who) * E + lane;
    m = 0.0;
    if (lane < E && e < p.V) m = token_mass<DT, ENS, NCH>(sh.kc, u, cf, inv, e);
    k = first_reach(m, scan(m, E), before, at);
    const int token = (step * 32 + who) * E + (k & 31);
    if (lane == 0 && k != -33) {
      p.out_tokens[u.uidx] = token;
      // Algorithm 2's Score returns the bonus token with its probability under the law it came from
      if (u.j == p.gamma && p.bonus_prob != nullptr) p.bonus_prob[u.b] = static_cast<float>(big_mass<DT, ENS, NCH>(sh.kc, u, inv, token));
    }
    return;
  }
}

// The block's position from the records of the streaming launch (and the row's outputs, see decide_row): every block decides
// its row for itself.  False when there is nothing to draw.
template <int DT, bool ENS, int NCH>
__device__ __forceinline__ bool decide_unit_to_draw(const KParams& p, DrawShared<NCH>& sh, RowShared& rs, int slot, int part) {
  const int tid = threadIdx.x;
  int b = slot, want = -1;
  if (p.draw_all) {
    const int drafts = p.B * p.gamma;  // every draft position, then the bonus positions
    b = slot < drafts ? slot / p.gamma : slot - drafts;
    want = slot < drafts ? slot % p.gamma : p.gamma;
  }
  DrawUnit<NCH>& u = sh.unit;
  decide_row<DT, ENS ? kEnsembleSample : kLogitSample>(
      p, rs, b, want,
      [&](const Finish& f, int j, unsigned word, int accepted, int drawable) {
        const int pi = proposer_of(p, b, j);
        const int pis = (pi >= 0 && pi < p.n) ? pi : 0;
        const int law = (j == p.gamma) ? (p.bonus_model >= 0 ? kDrawQ : kDrawR) : kDrawResidual;
        if (tid < NCH) {
          const bool live = tid < (ENS ? p.n : 2);
          u.nref[tid] = live ? -f.fsoft[tid].ref : 0.f;
          u.bt[tid] = live ? static_cast<float>(f.fsoft[tid].s * kBigShare) : INFINITY;
          u.ck[tid] = live ? coefficient<ENS>(p, tid, pis, law) * f.inv[tid] : 0.0;
          u.ct[tid] = static_cast<float>(u.ck[tid]);
        }
        if (tid == 0) {
          u.b = b;
          u.j = j;
          u.uidx = b * p.P + j;
          u.pis = pis;
          u.law = law;
          u.word = word;
          u.accepted = accepted;
          u.drawable = drawable;
          u.thr = (!ENS && p.mask_model >= 0) ? f.thr : -INFINITY;
          u.base = reinterpret_cast<const char*>(p.logits) +
                   (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
        }
      },
      [&](int a) { return part == 0 && (want < 0 || want == a); }, [&](int j) { return part == 0 && (want < 0 || want == j); });
  const bool emit = (rs.a == u.j);
  if (tid == 0) u.emit = emit ? 1 : 0;
  return u.drawable && (emit || u.j != p.gamma);
}

// One cluster of p.draw_parts blocks for each position.  All blocks of a cluster take the same way, and so meet at its barriers.
template <int DT, bool ENS, int NCH, bool AL>
__global__ void __launch_bounds__(NCH == 8 ? 256 : kMaxDrawThreads, NCH == 2 ? 2 : (NCH == 4 ? 1 : 2)) cos_draw_kernel(const __grid_constant__ KParams p) {
  extern __shared__ __align__(16) unsigned char draw_smem_raw[];
  DrawShared<NCH>& sh = *reinterpret_cast<DrawShared<NCH>*>(draw_smem_raw);
  double* slots = reinterpret_cast<double*>(draw_smem_raw + sizeof(DrawShared<NCH>));
  double* acc = slots + threadIdx.x;
  const int slot = blockIdx.x / p.draw_parts, rank = blockIdx.x % p.draw_parts, nw = blockDim.x >> 5;
  if (threadIdx.x < COS_MAX_MODELS) {
    DrawConst& kc = sh.kc;
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
  cluster_arrive();  // (the first block has begun: its shared memory may be written to)
  // launched while the kernel before it drains; nothing but inputs is read before that one is complete
  bool draws;
  if (NCH != 8 && p.decide) {
    RowShared& rs = *reinterpret_cast<RowShared*>(slots);
    draws = decide_unit_to_draw<DT, ENS, NCH>(p, sh, rs, slot, rank);
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    DrawUnit<NCH> d;
    draws = load_unit<DT, ENS, NCH>(p, slot, d);
    if (threadIdx.x == 0) sh.unit = d;
  }
  cluster_wait();
  if (!draws) return;
  __syncthreads();
  draw_sweep<DT, ENS, NCH, AL>(p, sh, rank * nw + (threadIdx.x >> 5), p.draw_parts * nw, acc);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cluster_arrive();
  cluster_wait();
  if (rank == 0) {
    __syncthreads();
    locate<DT, ENS, NCH, AL>(p, sh, acc);
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
