// The streaming launch of a run: every logit is read once (Eq. 3-5).
#ifndef COS_STREAM_CUH
#define COS_STREAM_CUH

#include "cos_common.cuh"

namespace cosv {

// Split: the positions' 16-byte vectors (the same vectors of all models of a position go together) form one line in the order of
// memory, cut into p.st_workers equal contiguous shares, one for each warp of a single wave of blocks.  So every warp streams the
// same number of bytes for any batch and vocabulary, with 4 KB in flight, and does nothing else: it leaves one record per model
// (partial softmax statistics or argmaxes) for every position it had a part of, and the next launch merges the records of a row's
// positions and decides (see cos_decide.cuh).  Where there are enough shares to a position they end where it ends, and short
// shares of an ensemble are one model's (see plan_line).  Models that agree at a position are cut at the same places, so that
// their statistics are the same bit for bit.
// What bounds it: HBM in large runs (256 rows of 256000 tokens, 2.36 GB: 355 us, 6.6 TB/s), in small ones the latency of one batch
// of loads and the launch (one row of 6 x 2 x 151936 entries: 4 us).
// Measured on 1152 rows of 151936 bf16 entries (350 MB): 60 us (5.8 TB/s); whole positions per block of 16 warps, as before, 65 to
// 70 us; shares of blocks instead of warps 65; 4 vectors in flight per lane 2 us more.  Reporting every part (fence, counter) cost
// 20 us more, deciding in the same launch another 17, the sweep in a function of its own 8; handing the last quarter out in
// items of 8 KB as warps become free 10 (each item pays a memory round trip and a record).
constexpr int kStreamThreads = 1024;  // most of a block: one per multiprocessor (64 registers)
constexpr int kStreamDepth = 8;      // vectors in flight per lane

struct Decision {  // one position's outcome
  int accept, status, cand;
  int natoms, drawable;
  int atom_tok[COS_MAX_MODELS];
  double atom_mass[COS_MAX_MODELS];
  double ratio, r_d, q_d, S;
  double prob;  // greedy, bonus position: probability of cand under the law it came from
};

struct Finish {  // what a position is decided from, and the decision
  union {
    SoftPart fsoft[COS_MAX_MODELS];  // merged statistics (sampling)
    ArgPart farg[COS_MAX_MODELS];    // merged argmaxes (greedy)
  };
  double pdraft[COS_MAX_MODELS];     // sampling: probability of the draft token under each softmax, NaN where its statistics are of no use
  float thr;                         // plausibility threshold (NaN: the gating model's logits hold one)
  Decision dec;
};

// x / d for places in the line (x < 2^53, quotient an int): a multiplication and a correction; the compiler's 64-bit division
// is 100 instructions long, and code is what the short launches spend their time on.
__device__ __forceinline__ int line_div(long long x, int d, double inv) {
  int q = static_cast<int>(static_cast<double>(x) * inv);
  const long long r = x - static_cast<long long>(q) * d;
  if (r < 0) --q;
  if (r >= d) ++q;
  return q;
}
__device__ __forceinline__ int worker_of(const KParams& p, long long x) { return line_div(x, p.st_share, p.st_inv_share); }
__device__ __forceinline__ long long worker_lo(const KParams& p, int w) {
  const long long x = static_cast<long long>(w) * p.st_share;
  return x < p.st_line ? x : p.st_line;
}

// Entries of a row that are not part of its whole vectors: [0, head) and [tail, V), fewer than three vectors in all.
struct Ragged {
  int head, tail;
};
template <int DT, bool AL>
__device__ __forceinline__ Ragged ragged_of(int V) {
  const VecRange w = whole_vectors<DT, AL>(V);
  Ragged r;
  r.head = w.hi > w.lo ? w.lo * Elem<DT>::E : 0;
  r.tail = w.hi > w.lo ? w.hi * Elem<DT>::E : 0;
  return r;
}
// The lane's entry of them, or -1.
__device__ __forceinline__ int ragged_entry(const Ragged& r, int V, int lane) {
  const int e = lane < r.head ? lane : r.tail + lane - r.head;
  return e < V ? e : -1;
}

__device__ __forceinline__ float max_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
template <int DT>
__device__ __forceinline__ unsigned max2_nan(unsigned a, unsigned b) {
  unsigned d;
  if (DT == COS_DTYPE_BF16)
    asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  else
    asm("max.NaN.f16x2 %0, %1, %2;" : "=r"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ float max3(float a, float b, float c) {  // (a NaN counts for nothing)
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// The largest entry of a vector, NaN if there is one; MAG: the largest magnitude.
template <int DT, bool MAG>
__device__ __forceinline__ float vector_max(const uint4& r) {
  if (DT == COS_DTYPE_F32) {
    const float a = __uint_as_float(r.x), b = __uint_as_float(r.y), c = __uint_as_float(r.z), d = __uint_as_float(r.w);
    return MAG ? max_nan(max_nan(fabsf(a), fabsf(b)), max_nan(fabsf(c), fabsf(d))) : max_nan(max_nan(a, b), max_nan(c, d));
  }
  const unsigned k = MAG ? 0x7fff7fffu : 0xffffffffu;
  const unsigned m = max2_nan<DT>(max2_nan<DT>(r.x & k, r.y & k), max2_nan<DT>(r.z & k, r.w & k));
  const uint4 q = make_uint4(m, 0u, 0u, 0u);
  return max_nan(entry<DT>(q, 0), entry<DT>(q, 1));
}

// Sums of a lane, two at a time: a few vectors plainly, then compensated (Kahan), every operation one packed instruction; so
// a share may be thousands of vectors long and its sum is as good as a short one's.
struct Comp2 {
  f32x2 sum, nc;  // running sum, minus the compensation
  __device__ __forceinline__ void init() { sum = nc = pack2(0.f, 0.f); }
  __device__ __forceinline__ void add(f32x2 v) {
    const f32x2 y = add2(v, nc);
    const f32x2 t = add2(sum, y);
    nc = add2(y, fma2(t, pack2(-1.f, -1.f), sum));
    sum = t;
  }
  __device__ __forceinline__ float total() const { return (lo2(sum) + hi2(sum)) + (lo2(nc) + hi2(nc)); }
};

// Reference exponent of a lane's sum: fixed, from its first vector, a whole number (sums with such references rescale exactly); 0 where
// that is not finite (see kTinySum).
__device__ __forceinline__ float seed_ref(float vmax, float c) {
  const float cand = vmax * c;
  return (fabsf(cand) < INFINITY) ? floorf(cand) : 0.f;
}

// sum of 2^(x c + nref) over one vector, in two halves
template <int DT>
__device__ __forceinline__ f32x2 vector_sum(const uint4& r, f32x2 c2, f32x2 nref2) {
  constexpr int H = Elem<DT>::E / 2;
  f32x2 x[H], s;
  unpack_pairs<DT>(r, x);
#pragma unroll
  for (int k = 0; k < H; ++k) {
    const f32x2 t = fma2(x[k], c2, nref2);
    const f32x2 e = pack2(ex2_approx(lo2(t)), ex2_approx(hi2(t)));
    s = k == 0 ? e : add2(s, e);
  }
  return s;
}

// The same segment with a running maximum, for the lane whose fixed reference did not hold.  Rare, but for logits of which most are
// -inf: four vectors at a time.
template <int DT, bool AL>
__device__ __noinline__ LaneSoft soft_online(const char* row, int v, int v1, float c) {
  LaneSoft acc;
  acc.init();
#pragma unroll 1
  for (; v < v1; v += 128) {
    uint4 raw[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      raw[u] = neg_inf_vector<DT>();
      if (v + u * 32 < v1) raw[u] = load_whole<DT, AL>(row, v + u * 32);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      float x[Elem<DT>::E];
      Elem<DT>::unpack(raw[u], x);
      acc.add_online(x, c);
    }
  }
  return acc;
}

// Softmax statistics of vectors [v0, v1) of one row and, with `ragged`, of its ragged entries; every lane's own part.
template <int DT, bool AL, bool LONG>
__device__ __forceinline__ LaneSoft soft_segment(const char* row, int v0, int v1, bool ragged, int V, float c) {
  constexpr int U = kStreamDepth;
  const int lane = threadIdx.x & 31;
  const f32x2 c2 = pack2(c, c);
  LaneSoft acc;
  acc.init();
  int v = v0 + lane;
  if (v < v1) {
    uint4 raw[U];
    Comp2 total;
    total.init();
    auto fetch = [&](int at, uint4& r) {
      r = neg_inf_vector<DT>();
      if (at < v1) r = load_whole<DT, AL>(row, at);
    };
    if (LONG) {
#pragma unroll
      for (int u = 0; u < U; ++u) fetch(v + u * 32, raw[u]);
      bool empty = true;
      for (; v < v1; v += U * 32) {
        if (empty) {  // (nothing but -inf so far, if anything: nothing was added)
          float m = vector_max<DT, false>(raw[0]);
          if (m == -INFINITY) {
#pragma unroll
            for (int u = 1; u < U; ++u) m = max_nan(m, vector_max<DT, false>(raw[u]));
          }
          empty = m == -INFINITY;
          acc.ref = empty ? -INFINITY : seed_ref(m, c);
        }
        const float n = empty ? 0.f : -acc.ref;
        const f32x2 nref2 = pack2(n, n);
        f32x2 s = pack2(0.f, 0.f);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          s = add2(s, vector_sum<DT>(raw[u], c2, nref2));
          fetch(v + (U + u) * 32, raw[u]);
        }
        total.add(s);
      }
    } else {
      f32x2 nref2 = pack2(0.f, 0.f);
      bool first = true;
      for (; v < v1; v += U * 32) {
#pragma unroll
        for (int u = 0; u < U; ++u) fetch(v + u * 32, raw[u]);
        if (first) {
          acc.ref = seed_ref(vector_max<DT, false>(raw[0]), c);
          nref2 = pack2(-acc.ref, -acc.ref);
          first = false;
        }
        f32x2 s = vector_sum<DT>(raw[0], c2, nref2);
#pragma unroll
        for (int u = 1; u < U; ++u) s = add2(s, vector_sum<DT>(raw[u], c2, nref2));
        total.add(s);
      }
    }
    acc.s = total.total();
    if (!acc.holds()) acc = soft_online<DT, AL>(row, v0 + lane, v1, c);
  }
  if (ragged) {
    const int e = ragged_entry(ragged_of<DT, AL>(V), V, lane);
    if (e >= 0) acc.add_online1(Elem<DT>::load1(row, e), c);
  }
  return acc;
}

// Argmax of vectors [v0, v1) of one row (lowest index among equals) and whether a NaN or +inf was seen; the warp's result.
template <int DT, bool AL>
__device__ __forceinline__ ArgPart arg_segment(const char* row, int v0, int v1, bool ragged, int V) {
  constexpr int U = kStreamDepth, E = Elem<DT>::E;
  const int lane = threadIdx.x & 31;
  float best = -INFINITY;  // (sticks at NaN)
  int bestv = -1;
  for (int v = v0 + lane; v < v1; v += U * 32) {
    uint4 raw[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      raw[u] = neg_inf_vector<DT>();
      if (v + u * 32 < v1) raw[u] = load_whole<DT, AL>(row, v + u * 32);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float m = vector_max<DT, false>(raw[u]);
      if (m > best) bestv = v + u * 32;
      best = max_nan(best, m);
    }
  }
  int idx = kNoReject, bad = !(best < INFINITY);
  if (bestv >= 0) {
    const uint4 r = load_whole<DT, AL>(row, bestv);
#pragma unroll
    for (int k = E - 1; k >= 0; --k)
      if (entry<DT>(r, k) == best) idx = bestv * E + k;
  }
  if (ragged) {
    const int e = ragged_entry(ragged_of<DT, AL>(V), V, lane);
    if (e >= 0) {
      const float x = Elem<DT>::load1(row, e);
      bad |= !(x < INFINITY);
      if (arg_better(x, e, best, idx)) {
        best = x;
        idx = e;
      }
    }
  }
  return warp_reduce_arg(static_cast<double>(best), idx, bad, lane);
}

struct LaneSoft2 {
  LaneSoft q, c;
};
// Tokens [e, end) one by one, running maximum: the ragged ends, and the lane whose fixed references did not hold.
template <int DT>
__device__ __noinline__ LaneSoft2 logit_online(const KParams& p, const char* base, int pis, float thr, int e, int end, LaneSoft2 a) {
  for (; e < end; ++e) {
    float cmb = 0.f, xq = -INFINITY, xe = 0.f;
    for (int i = 0; i < p.n; ++i) {
      const float x = Elem<DT>::load1(base + i * p.s_model * Elem<DT>::bytes, e);
      cmb = fmaf(p.w[i], x, cmb);
      if (i == pis) xq = x;
      if (i == p.mask_model) xe = x;
    }
    if (p.mask_model >= 0 && !(xe >= thr)) cmb = -INFINITY;
    a.q.add_online1(xq, p.cT);
    a.c.add_online1(cmb, p.cT);
  }
  return a;
}

// Softmax statistics of the proposer's logits and of the combined ones over vectors [v0, v1) of a position, four vectors of
// the first two models in flight (further models are read as they are needed).
// PAIR: exactly two models; MASKED: with the plausibility mask.
template <int DT, bool AL, bool PAIR, bool MASKED>
__device__ __forceinline__ LaneSoft2 logit_segment(const KParams& p, const char* base, long long row_step, LogitWeights lw, float cT,
                                                int v0, int v1, bool ragged) {
  constexpr int U = kStreamDepth / 2, H = Elem<DT>::E / 2;
  const int lane = threadIdx.x & 31;
  const bool pair = PAIR || p.n >= 2;
  const f32x2 c2 = pack2(cT, cT);
  LaneSoft2 acc;
  LaneSoft &accq = acc.q, &accc = acc.c;
  accq.init();
  accc.init();
  int v = v0 + lane;
  if (v < v1) {
    Comp2 tq, tc;
    tq.init();
    tc.init();
    f32x2 nq = pack2(0.f, 0.f), nc = nq;
    bool first = true;
    float top = -INFINITY;  // with a mask: whether the lane has a token that counts
    for (; v < v1; v += U * 32) {
      uint4 r0[U], r1[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        r0[u] = r1[u] = neg_inf_vector<DT>();
        if (v + u * 32 < v1) {
          r0[u] = load_whole<DT, AL>(base, v + u * 32);
          if (pair) r1[u] = load_whole<DT, AL>(base + row_step, v + u * 32);
        }
      }
      f32x2 sq = pack2(0.f, 0.f), sc = sq;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        f32x2 xq[H], cmb[H];
        const bool in = u == 0 || v + u * 32 < v1;
        logit_args<DT, PAIR, MASKED>(p, lw, r0[u], r1[u],
                                     [&](int i) {
                                       uint4 r = neg_inf_vector<DT>();
                                       if (in) r = load_whole<DT, AL>(base + i * row_step, v + u * 32);
                                       return r;
                                     },
                                     xq, cmb);
        if (u == 0 && first) {
          float mq = -INFINITY, mc = -INFINITY;
#pragma unroll
          for (int k = 0; k < H; ++k) {
            mq = fmaxf(mq, fmaxf(lo2(xq[k]), hi2(xq[k])));
            mc = fmaxf(mc, fmaxf(lo2(cmb[k]), hi2(cmb[k])));
          }
          accq.ref = seed_ref(mq, cT);
          accc.ref = seed_ref(mc, cT);
          nq = pack2(-accq.ref, -accq.ref);
          nc = pack2(-accc.ref, -accc.ref);
          first = false;
        }
        if (MASKED) {
#pragma unroll
          for (int k = 0; k < H; ++k) top = max3(top, lo2(cmb[k]), hi2(cmb[k]));
        }
        f32x2 vq = pack2(0.f, 0.f), vc = vq;
#pragma unroll
        for (int k = 0; k < H; ++k) {
          const f32x2 aq = fma2(xq[k], c2, nq), ac = fma2(cmb[k], c2, nc);
          vq = add2(vq, pack2(ex2_approx(lo2(aq)), ex2_approx(hi2(aq))));
          vc = add2(vc, pack2(ex2_approx(lo2(ac)), ex2_approx(hi2(ac))));
        }
        if (in) {  // (a vector that is not there could combine to anything)
          sq = add2(sq, vq);
          sc = add2(sc, vc);
        }
      }
      tq.add(sq);
      tc.add(sc);
    }
    accq.s = tq.total();
    accc.s = tc.total();
    if (MASKED && top == -INFINITY) accc.ref = -INFINITY;  // (the sum is 0, or NaN: a token inside the mask that is no number)
  }
  if (!accq.holds() || !accc.holds()) {  // rare
    accq.init();
    accc.init();
    for (v = v0 + lane; v < v1; v += 32) acc = logit_online<DT>(p, base, lw.pis, lw.thr, v * Elem<DT>::E, (v + 1) * Elem<DT>::E, acc);
  }
  if (ragged) {
    const int e = ragged_entry(ragged_of<DT, AL>(p.V), p.V, lane);
    if (e >= 0) acc = logit_online<DT>(p, base, lw.pis, lw.thr, e, e + 1, acc);
  }
  return acc;
}

// The argmax of the combined logits must be the fp64 one (the same chain of fused multiply-adds on every token, lowest index
// among equals).  A vector gets its largest fp32 value and a bound on the distance of any of its fp32 values from the
// fp64 ones, n 2^-23 sum_i |w_i| max |l_i|; the warp's largest value less its bound is below the maximum for certain, and
// only vectors that could reach it are evaluated in fp64, one or two of a batch, a token a lane.  (A bound for every token
// cost 5 instructions more for each logit: 564 us instead of 418 for 2304 positions of two 256000-token models.  Without a bound to
// start from every first vector was evaluated, each by its lane: one row of 32000 tokens took 21.4 us on the device, with it 7.6;
// 64 rows of 256000 with a mask 309 and 93.)
struct ArgPart2 {
  ArgPart q, c;
};
__device__ __forceinline__ float warp_max(float x) {  // (floats ordered as unsigned integers; no NaN)
  const unsigned bits = __float_as_uint(x);
  const unsigned top = __reduce_max_sync(0xffffffffu, bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u));
  return __uint_as_float(top ^ ((top >> 31) ? 0x80000000u : 0xffffffffu));
}
template <int DT, bool AL, bool PAIR, bool MASKED>
__device__ __forceinline__ ArgPart2 logit_arg_segment(const KParams& p, const char* base, long long row_step, LogitWeights lw, int v0,
                                                   int v1, bool ragged) {
  constexpr int U = kStreamDepth / 2, E = Elem<DT>::E, H = E / 2, G = 32 / E;
  const int lane = threadIdx.x & 31;
  const bool pair = PAIR || p.n >= 2;
  const int pis = lw.pis;
  const float slack = static_cast<float>(PAIR ? 2 : p.n) * 1.1920929e-07f;  // n * 2^-23
  const float wa0 = fabsf(lw.w0), wa1 = pair ? fabsf(lw.w1) : 0.f;
  double best = -INFINITY;
  int idx = kNoReject, bad = 0;
  float lo = -INFINITY, qbest = -INFINITY;  // lo: below the maximum, the same for the whole warp
  int qv = -1;
  auto consider = [&](int e) {
    double cm = 0.0;
    float gate = 0.f;
    const int n = PAIR ? 2 : p.n;
#pragma unroll 2
    for (int i = 0; i < n; ++i) {
      const float x = Elem<DT>::load1(base + i * row_step, e);
      bad |= !(x < INFINITY);
      cm = fma(p.w64[i], static_cast<double>(x), cm);
      if (MASKED && i == lw.mask_model) gate = x;
    }
    const bool in = !MASKED || gate >= lw.thr;
    bad |= (in && cm != cm);
    if (in && arg_better(cm, e, best, idx)) {
      best = cm;
      idx = e;
    }
  };
  for (int vb = v0; vb < v1; vb += U * 32) {  // (a warp goes through the loop as one)
    const int v = vb + lane;
    uint4 r0[U], r1[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      r0[u] = r1[u] = neg_inf_vector<DT>();
      if (v + u * 32 < v1) {
        r0[u] = load_whole<DT, AL>(base, v + u * 32);
        if (pair) r1[u] = load_whole<DT, AL>(base + row_step, v + u * 32);
      }
    }
    float hi[U], low = -INFINITY;  // no value of the vector is above hi; some value of the lane's is not below low
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int vu = v + u * 32;
      const bool there = vu < v1;
      float bound = wa0 * vector_max<DT, true>(r0[u]);
      if (pair) bound = fmaf(wa1, vector_max<DT, true>(r1[u]), bound);
      uint4 rq = pick_vector(pis == 0, r0[u], r1[u]);
      f32x2 xq[H], cmb[H];
      logit_args<DT, PAIR, MASKED>(p, lw, r0[u], r1[u],
                                   [&](int i) {
                                     uint4 r = neg_inf_vector<DT>();
                                     if (there) r = load_whole<DT, AL>(base + i * row_step, vu);
                                     if (i == pis) rq = r;
                                     bound = fmaf(fabsf(p.w[i]), vector_max<DT, true>(r), bound);
                                     return r;
                                   },
                                   xq, cmb);
      const float mq = vector_max<DT, false>(rq);
      if (mq > qbest) {
        qbest = mq;
        qv = vu;
      }
      float mc = -INFINITY;
#pragma unroll
      for (int k = 0; k < H; ++k) mc = max3(mc, lo2(cmb[k]), hi2(cmb[k]));
      const bool sound = bound < INFINITY;  // (a NaN or an infinity among the logits has to be looked at)
      hi[u] = !there ? -INFINITY : (sound ? __fmaf_ru(bound, slack, mc) : INFINITY);
      if (there && sound) low = fmaxf(low, __fmaf_rd(-bound, slack, mc));
    }
    lo = fmaxf(lo, warp_max(low));
    unsigned reach = 0u;  // (-inf: no token of the vector counts)
#pragma unroll
    for (int u = 0; u < U; ++u) reach |= (hi[u] >= lo && hi[u] > -INFINITY) ? 1u << u : 0u;
    unsigned any = __reduce_or_sync(0xffffffffu, reach);
    if (any) {
#pragma unroll 1
      for (; any; any &= any - 1) {
        const int u = __ffs(any) - 1;
        unsigned m = __ballot_sync(0xffffffffu, (reach >> u) & 1u);
#pragma unroll 1
        while (m) {
          unsigned t = m;
#pragma unroll
          for (int q = 0; q < G; ++q) {
            if (q < lane / E) t &= t - 1;
            m &= m - 1;
          }
          if (t) consider((vb + u * 32 + __ffs(t) - 1) * E + lane % E);
        }
      }
      lo = fmaxf(lo, warp_max(__double2float_rd(best)));
    }
  }
  int qidx = kNoReject;
  if (qv >= 0) {
    const uint4 r = load_whole<DT, AL>(base + pis * row_step, qv);
#pragma unroll
    for (int k = E - 1; k >= 0; --k)
      if (entry<DT>(r, k) == qbest) qidx = qv * E + k;
  }
  if (ragged) {
    const int e = ragged_entry(ragged_of<DT, AL>(p.V), p.V, lane);
    if (e >= 0) {
      consider(e);
      const float x = Elem<DT>::load1(base + pis * row_step, e);
      if (arg_better(x, e, qbest, qidx)) {
        qbest = x;
        qidx = e;
      }
    }
  }
  ArgPart2 out;
  out.q = warp_reduce_arg(static_cast<double>(qbest), qidx, bad, lane);
  out.c = warp_reduce_arg(best, idx, bad, lane);
  return out;
}

// ------------------------------------------------------------------------------------
// publishing a unit and the per-row first-rejection scan (Sec. 3.1)
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void push_job(const KParams& p, int idx, int emit) {
  const int k = atomicAdd(p.job_count, 1);
  if (k < p.max_jobs) p.jobs[k] = make_int2(idx, emit);
}

// Record a unit's decision; the last unit of a row to arrive scans for the first
// rejection, writes the row's outputs and, where a token has to be drawn, names that position
// for the drawing launch (which fills in out_tokens[b][a]).
// `word4`: sampling modes: whether a token can be drawn at this unit; greedy modes: the bits of the bonus
// token's probability (a float), NaN away from the bonus position.
__device__ __forceinline__ void publish_unit(const KParams& p, int b, int j, int accept, int status, int cand, int word4,
                             double ratio, double r_d, double q_d, double S) {
  const int idx = b * p.P + j;
  if (p.diag) {
    float* d = p.diag + static_cast<long long>(idx) * 4;
    d[0] = static_cast<float>(ratio);
    d[1] = static_cast<float>(r_d);
    d[2] = static_cast<float>(q_d);
    d[3] = static_cast<float>(S);
  }
  int4 res = make_int4(accept, status, cand, word4);
  __stcg(&p.unit_res[idx], res);
  if (p.early_exit && !accept && j < p.gamma) atomicMin(&p.row_reject[b], j);  // later positions may be left unread
  __threadfence();
  // The row's word counts its published positions (low six bits) and, for rows of up to kPackedP positions,
  // also carries one "not accepted" bit and one "has status bits" bit per position: the last position to
  // arrive then knows the first rejection from the value the atomic returns, without reading the others.
  const bool packed = (p.P <= kPackedP);
  int mine = 1;
  if (packed) {
    if (!accept || j == p.gamma) mine |= 1 << (6 + j);
    if (status) mine |= 1 << (6 + kPackedP + j);
  }
  const int prev = atomicAdd(&p.row_arrivals[b], mine);
  if ((packed ? (prev & 63) : prev) != p.P - 1) return;  // longer rows keep a plain count in the word
  // last unit of the row: every other unit's result is visible after the fence below
  __threadfence();
  int a = p.gamma;
  unsigned st = 0;
  int tok = -1, draw = 0;
  if (packed) {
    const int total = prev + mine;  // every position added its own bits once: no carries
    a = __ffs((total >> 6) & ((1 << kPackedP) - 1)) - 1;
    const int4 u = __ldcg(&p.unit_res[b * p.P + a]);
    tok = u.z;
    draw = u.w;
    int with_status = (total >> (6 + kPackedP)) & ((2 << a) - 1);
    while (with_status) {  // rare: some position up to the first rejection reported status bits
      const int k = __ffs(with_status) - 1;
      with_status &= with_status - 1;
      st |= static_cast<unsigned>(__ldcg(&p.unit_res[b * p.P + k]).y);
    }
  } else {
    for (int k = 0; k < p.P; ++k) {
      int4 u = __ldcg(&p.unit_res[b * p.P + k]);
      st |= static_cast<unsigned>(u.y);
      if (k == p.gamma || !u.x) {
        a = k;
        tok = u.z;
        draw = u.w;
        break;
      }
    }
  }
  if (p.bonus_prob != nullptr) {
    // sampling modes: the drawing launch fills it in after a full acceptance; greedy modes know it here
    const bool known = p.greedy && a == p.gamma && tok >= 0;
    p.bonus_prob[b] = known ? __int_as_float(draw) : __int_as_float(0x7fc00000);
  }
  if (p.greedy) draw = 0;
  p.accept_count[b] = a;
  int* o = p.out_tokens + static_cast<long long>(b) * p.P;
  for (int k = 0; k < p.P; ++k) o[k] = (k < a) ? p.drafts[b * p.gamma + k] : (k == a ? tok : -1);
  p.row_status[b] = st;
  p.row_arrivals[b] = 0;  // leave the scratch ready for the next run
  if (p.early_exit) p.row_reject[b] = kNoReject;
  if (!p.greedy) p.row_draw[b] = draw ? a : -1;
  if (draw && p.use_jobs) push_job(p, b * p.P + a, 1);
}

// The accept test of one (row, position) from the merged statistics (Eq. 6), taken by one thread in fp64; greedy modes also
// settle the replacement token here.  Reads fsoft / farg / pdraft / thr, writes d.  (Logit-level greedy: farg[0] is the
// proposer's argmax, farg[1] the combined one.)
template <int DT, int MODE>
__device__ __forceinline__ void decide_unit(const KParams& p, const Finish& sh, Decision& d, double u_acc, double u_smp, bool is_bonus, int draft, bool draft_ok,
                                            int pi, bool pi_ok, int pis) {
  const bool mask_bad = MODE == kLogitGreedy && p.mask_model >= 0 && sh.thr != sh.thr;
  constexpr bool kSample = (MODE == kEnsembleSample || MODE == kLogitSample);
  const double kNaN = __longlong_as_double(0x7ff8000000000000LL);
  const double kInf = __longlong_as_double(0x7ff0000000000000LL);
  d.accept = 0;
  d.status = 0;
  d.cand = -1;
  d.natoms = 0;
  d.ratio = d.r_d = d.q_d = d.S = d.prob = kNaN;
  bool finite = pi_ok;
  if (kSample) {
    double r_d = 0.0, q_d;
    if (MODE == kEnsembleSample) {
#pragma unroll 1
      for (int i = 0; i < p.n; ++i) r_d += p.w64[i] * sh.pdraft[i];
      q_d = sh.pdraft[pis];
    } else {
      q_d = sh.pdraft[0];
      r_d = sh.pdraft[1];
    }
    finite = finite && r_d == r_d && q_d == q_d;
    if (!finite) {
      d.status |= COS_ROW_NONFINITE;
    } else if (!is_bonus) {
      if (draft_ok) {
        d.r_d = r_d;
        d.q_d = q_d;
        if (q_d > 0.0) {
          d.ratio = r_d / q_d;
        } else {
          d.status |= COS_ROW_Q_ZERO;
          d.ratio = (r_d > 0.0) ? kInf : 0.0;
        }
        d.accept = accepts(u_acc, r_d, q_d) ? 1 : 0;
      } else {
        d.status |= COS_ROW_BAD_DRAFT;
      }
    }
  } else {
    // greedy: distributions are atoms at lowest-index argmaxes
    int qtok;
    if (MODE == kEnsembleGreedy) {
#pragma unroll 1
      for (int i = 0; i < p.n; ++i) finite = finite && !sh.farg[i].bad && isfinite(sh.farg[i].val);
      qtok = sh.farg[pis].idx;
    } else {
      finite = finite && !sh.farg[0].bad && !sh.farg[1].bad && isfinite(sh.farg[0].val) && isfinite(sh.farg[1].val);
      if (mask_bad) finite = false;
      qtok = sh.farg[0].idx;
    }
    if (!finite) {
      d.status |= COS_ROW_NONFINITE;
    } else {
      // atoms of r, sorted by token, masses accumulated in model order
      if (MODE == kEnsembleGreedy) {
#pragma unroll 1
        for (int i = 0; i < p.n; ++i) {
          int t = sh.farg[i].idx, pos = 0;
#pragma unroll 1
          while (pos < d.natoms && d.atom_tok[pos] < t) ++pos;
          if (pos < d.natoms && d.atom_tok[pos] == t) {
            d.atom_mass[pos] += p.w64[i];
          } else {
#pragma unroll 1
            for (int k = d.natoms; k > pos; --k) {
              d.atom_tok[k] = d.atom_tok[k - 1];
              d.atom_mass[k] = d.atom_mass[k - 1];
            }
            d.atom_tok[pos] = t;
            d.atom_mass[pos] = 0.0 + p.w64[i];
            ++d.natoms;
          }
        }
      } else {
        d.natoms = 1;
        d.atom_tok[0] = sh.farg[1].idx;
        d.atom_mass[0] = 1.0;
      }
      auto r_at = [&](int t) {
#pragma unroll 1
        for (int k = 0; k < d.natoms; ++k)
          if (d.atom_tok[k] == t) return d.atom_mass[k];
        return 0.0;
      };
      bool use_r = is_bonus;
      if (!is_bonus) {
        if (draft_ok) {
          d.r_d = r_at(draft);
          d.q_d = (draft == qtok) ? 1.0 : 0.0;
          if (d.q_d > 0.0) {
            d.ratio = d.r_d / d.q_d;
          } else {
            d.status |= COS_ROW_Q_ZERO;
            d.ratio = (d.r_d > 0.0) ? kInf : 0.0;
          }
          d.accept = (u_acc <= fmin(1.0, d.ratio)) ? 1 : 0;
        } else {
          d.status |= COS_ROW_BAD_DRAFT;
        }
        // residual max(0, r - q) over the atoms, summed in token order
        double S = 0.0;
#pragma unroll 1
        for (int k = 0; k < d.natoms; ++k) S += fmax(0.0, d.atom_mass[k] - (d.atom_tok[k] == qtok ? 1.0 : 0.0));
        d.S = S;
        if (!(S > 0.0)) {
          use_r = true;
          if (!d.accept) d.status |= COS_ROW_RESIDUAL_EMPTY;
        }
      }
      // inverse CDF over the atoms (token order): smallest k with running sum >= u * total
      double total = 0.0;
#pragma unroll 1
      for (int k = 0; k < d.natoms; ++k)
        total += use_r ? d.atom_mass[k] : fmax(0.0, d.atom_mass[k] - (d.atom_tok[k] == qtok ? 1.0 : 0.0));
      const double target = u_smp * total;
      double run = 0.0;
      int lastpos = -1;
      d.cand = -1;
#pragma unroll 1
      for (int k = 0; k < d.natoms; ++k) {
        double m = use_r ? d.atom_mass[k] : fmax(0.0, d.atom_mass[k] - (d.atom_tok[k] == qtok ? 1.0 : 0.0));
        run += m;
        if (m > 0.0) lastpos = d.atom_tok[k];
        if (d.cand < 0 && m > 0.0 && run >= target) d.cand = d.atom_tok[k];
      }
      if (d.cand < 0) d.cand = lastpos;
      if (is_bonus) {
        if (p.bonus_model >= 0) {  // the named model's one-hot law (its argmax sits in the proposer's slot)
          d.cand = qtok;
          d.prob = 1.0;
        } else {
          d.prob = r_at(d.cand);
        }
      }
    }
  }
  d.drawable = (kSample && finite) ? 1 : 0;
}

// Rescale a sum from reference exponent `ref` to R >= ref: an exact power of two where the references are whole numbers (sums
// whose fixed reference did not hold have others).
static __device__ __noinline__ double rescale_any(double s, float ref, float R) {
  return s == 0.0 ? 0.0 : s * exp2(static_cast<double>(ref) - static_cast<double>(R));
}
__device__ __forceinline__ double rescale(double s, float ref, float R) {
  const float d = fmaxf(ref - R, -1000.f);  // (a sum that far below is nothing; the empty sum's reference is minus infinity)
  if (d != floorf(d)) return rescale_any(s, ref, R);
  return s * __hiloint2double((1023 + static_cast<int>(d)) << 20, 0);
}

// The records of the line: `slots` (a model each, or the proposer's and the combined logits) for every position r that share w
// has a part of; the pairs (r, w) follow one another with r + w rising.
template <int MODE>
__device__ __forceinline__ int record_slots(const KParams& p) {
  return (MODE == kEnsembleSample || MODE == kEnsembleGreedy) ? p.n : 2;
}
// Where the records of position j of row b are: `count` times `slots` of them.
struct RecordRange {
  const int4* first;
  int count;
};
template <int MODE>
__device__ __forceinline__ RecordRange records_of(const KParams& p, int b, int j) {
  const int slots = record_slots<MODE>(p);
  // (where every row has a line of its own, the records of a row follow those of the row before)
  const long long at = static_cast<long long>(p.st_row ? j : b * p.P + j) * p.st_nv;
  const int w0 = worker_of(p, at), w1 = worker_of(p, at + p.st_nv - 1);
  RecordRange q;
  q.first = p.st_rec + (static_cast<size_t>(b) * (p.P + p.st_row) + j + w0) * slots;
  q.count = w1 - w0 + 1;
  return q;
}

// Merge slot i of a position over its records; `g` lanes (a power of two, aligned) share the work, `sub` is the lane's place
// among them.  Every lane of the warp calls this (one with an empty range only takes part in the exchanges).  All lanes of a
// group get the sums, the first one of them argmaxes.  `AT` records at a time are on their way, and every sum is rescaled once, to the
// reference of the whole group: one record after another took 10 us for the 148 of each position of a 6-position row.  Sums four at a time
// where a block of 512 threads leaves a pair more lanes than that many trips need, otherwise eight (in the deciding launch, whose groups are of a
// few lanes, one row of 5 x 8 x 128256 fp32 takes 58.3 us with four and 53.8 with eight, of 5 x 5 x 128256 50.4 and 49.0); argmaxes are
// compared one after the other, so that fewer trips count for more.
struct Merged {
  SoftPart soft;
  ArgPart arg;
  float thr;
};
template <int MODE, int AT>
__device__ __forceinline__ Merged merge_slot(const KParams& p, const RecordRange& q, int i, int g, int sub) {
  constexpr bool kSample = (MODE == kEnsembleSample || MODE == kLogitSample);
  constexpr int kAtOnce = AT;
  const int slots = record_slots<MODE>(p);
  Merged m;
  m.soft.ref = -INFINITY;
  m.soft.s = 0.0;
  m.arg.val = -INFINITY;
  m.arg.idx = kNoReject;
  m.arg.bad = 0;
  m.thr = -INFINITY;
  int4 v4[kAtOnce];
  auto fetch = [&](int c0) {
#pragma unroll
    for (int k = 0; k < kAtOnce; ++k) {
      const int c = c0 + k * g;
      v4[k] = make_int4(0, kSample ? 0 : static_cast<int>(0xfff00000u), kSample ? static_cast<int>(0xff800000u) : kNoReject, 0);
      if (c < q.count) v4[k] = __ldcg(q.first + static_cast<size_t>(c) * slots + i);
    }
  };
  if (kSample) {
    fetch(sub);
    if (sub < q.count) m.thr = __int_as_float(v4[0].w);
#pragma unroll 1
    for (int c0 = sub;;) {
      float top = m.soft.ref;
#pragma unroll
      for (int k = 0; k < kAtOnce; ++k) top = fmaxf(top, __int_as_float(v4[k].z));
      const bool more = __any_sync(0xffffffffu, c0 + kAtOnce * g < q.count);
      if (!more) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1)
          if (d < g) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, d));
      }
      double s = c0 == sub ? 0.0 : rescale(m.soft.s, m.soft.ref, top);
#pragma unroll
      for (int k = 0; k < kAtOnce; ++k) s += rescale(__hiloint2double(v4[k].y, v4[k].x), __int_as_float(v4[k].z), top);
      m.soft.s = s;
      m.soft.ref = top;
      if (!more) break;
      c0 += kAtOnce * g;
      fetch(c0);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1)
      if (d < g) m.soft.s += __shfl_xor_sync(0xffffffffu, m.soft.s, d);
  } else {
    for (int c0 = sub; c0 < q.count; c0 += kAtOnce * g) {
      fetch(c0);
#pragma unroll
      for (int k = 0; k < kAtOnce; ++k) {
        const double v = __hiloint2double(v4[k].y, v4[k].x);
        m.arg.bad |= v4[k].w & 1;
        if (v4[k].w & 2) m.thr = __int_as_float(0x7fc00000);
        if (arg_better(v, v4[k].z, m.arg.val, m.arg.idx)) {
          m.arg.val = v;
          m.arg.idx = v4[k].z;
        }
      }
    }
    for (int d = g / 2; d > 0; d >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, m.arg.val, d);
      const int oi = __shfl_xor_sync(0xffffffffu, m.arg.idx, d);
      m.arg.bad |= __shfl_xor_sync(0xffffffffu, m.arg.bad, d);
      if (arg_better(ov, oi, m.arg.val, m.arg.idx)) {
        m.arg.val = ov;
        m.arg.idx = oi;
      }
    }
  }
  return m;
}

// The plausibility threshold of a position from the largest logit of the gating model (key of the mask launch); NaN where
// that model's logits hold one.
__device__ __forceinline__ float mask_bound(const KParams& p, unsigned key) {
  if (key > 0xff800000u) return __int_as_float(0x7fc00000);
  const float top = __uint_as_float(key ^ ((key >> 31) ? 0x80000000u : 0xffffffffu));
  // l >= max + ln(alpha) in fp64 is the same as l >= (that bound rounded up to fp32) for fp32 l
  return __double2float_ru(static_cast<double>(top) + p.ln_alpha);
}

// Probability of the draft token under softmax i, with the constant the sweep used: what it needs of the logits (fetched, and combined,
// before the statistics are there; nothing where draft < 0), and the rest once they are merged.
struct DraftLogit {
  double x;    // the softmax's logit
  float gate;  // what the plausibility threshold is compared with
};
template <int DT, int MODE>
__device__ __forceinline__ DraftLogit draft_logit(const KParams& p, const char* base, int i, int pis, int draft) {
  DraftLogit d = {0.0, 0.f};
  if (draft < 0) return d;
  const long long row_step = p.s_model * Elem<DT>::bytes;
  if (MODE == kEnsembleSample || i == 0) {
    d.x = static_cast<double>(Elem<DT>::load1(base + (MODE == kEnsembleSample ? i : pis) * row_step, draft));
  } else {
#pragma unroll 2
    for (int k = 0; k < p.n; ++k) {
      const float l = Elem<DT>::load1(base + k * row_step, draft);
      d.x = k == 0 ? p.w64[0] * static_cast<double>(l) : fma(p.w64[k], static_cast<double>(l), d.x);
      if (k == p.mask_model) d.gate = l;
    }
  }
  return d;
}
// NaN where the statistics, or the threshold, are of no use.
template <int MODE>
__device__ __forceinline__ double draft_probability(const KParams& p, const DraftLogit& d, int i, int draft, float thr, const SoftPart& f, double inv) {
  const double nan = __longlong_as_double(0x7ff8000000000000LL);
  if (!(isfinite(f.ref) && isfinite(f.s) && f.s > 0.0)) return nan;
  if (MODE == kLogitSample && p.mask_model >= 0) {
    if (thr != thr) return nan;
    if (i == 1 && !(d.gate >= thr)) return 0.0;
  }
  return draft < 0 ? 0.0 : exp2(d.x * p.cT64 - static_cast<double>(f.ref)) * inv;
}

// Largest logit of the gating model at every position, for the plausibility mask: the same split, over that model's rows
// alone.  (Positions need it before they can be swept, and the warps of the streaming launch do not wait for each other.)
template <int DT, bool AL>
__global__ void __launch_bounds__(kStreamThreads, 1) cos_mask_kernel(const __grid_constant__ KParams p) {
  constexpr int U = kStreamDepth;
  const int lane = threadIdx.x & 31;
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (w >= p.st_workers) return;
  const int v_lo = whole_vectors<DT, AL>(p.V).lo, v_hi = whole_vectors<DT, AL>(p.V).hi;
  for (long long x = worker_lo(p, w), end = worker_lo(p, w + 1); x < end;) {
    const int unit = line_div(x, p.st_nv, p.st_inv_nv);
    const int o0 = static_cast<int>(x - static_cast<long long>(unit) * p.st_nv);
    const int o1 = end - x < p.st_nv - o0 ? o0 + static_cast<int>(end - x) : p.st_nv;
    const int b = unit / p.P, j = unit % p.P;
    const char* row = reinterpret_cast<const char*>(p.logits) +
                      (p.mask_model * p.s_model + static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
    float best = -INFINITY;
    const int v1 = v_lo + o1 < v_hi ? v_lo + o1 : v_hi;
    for (int v = v_lo + o0 + lane; v < v1; v += U * 32) {
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
    if (lane == 0) atomicMax(&p.mask_key[unit], top);
    x += o1 - o0;
  }
}

__device__ __forceinline__ int4 pack_soft(const LaneSoft& a, float thr) {
  float R;
  const double s = static_cast<double>(warp_sum_soft(a, R));
  return make_int4(__double2loint(s), __double2hiint(s), __float_as_int(R), __float_as_int(thr));
}
__device__ __forceinline__ int4 pack_arg(const ArgPart& a, float thr) {
  return make_int4(__double2loint(a.val), __double2hiint(a.val), a.idx, a.bad | (thr != thr ? 2 : 0));
}

// The part of one position, vectors [o0, o1) of every model (ensembles: of models [i0, i1)), that lies in a warp's share: its records (lane 0 writes them).
// `settled`: the inputs may be read before the kernel ahead in the stream is complete; this waits for it before it writes.
template <int DT, int MODE, bool AL, bool PAIR, bool MASKED>
__device__ __forceinline__ void sweep_part(const KParams& p, const char* base, int o0, int o1, int i0, int i1, int pis, float thr, int4* rec,
                                           bool& waited) {
  const int lane = threadIdx.x & 31;
  const VecRange whole = whole_vectors<DT, AL>(p.V);
  const int v0 = whole.lo + o0, v1 = whole.lo + o1 < whole.hi ? whole.lo + o1 : whole.hi;
  const bool ragged = (o1 == p.st_nv);
  const long long row_step = p.s_model * Elem<DT>::bytes;
  auto put = [&](int i, const int4& v) {
    if (!waited) {
      asm volatile("griddepcontrol.wait;" ::: "memory");  // from here on as in an ordinary run
      waited = true;
    }
    if (lane == 0) __stcg(rec + i, v);
  };
  if (MODE == kEnsembleSample) {
    for (int i = i0; i < i1; ++i) put(i, pack_soft(soft_segment<DT, AL, PAIR>(base + i * row_step, v0, v1, ragged, p.V, p.cT), thr));
  } else if (MODE == kEnsembleGreedy) {
    for (int i = i0; i < i1; ++i) put(i, pack_arg(arg_segment<DT, AL>(base + i * row_step, v0, v1, ragged, p.V), thr));
  } else if (MODE == kLogitSample) {
    LaneSoft2 a;
    // (with a mask, which of two vectors is the proposer's is known to the code, not chosen entry by entry: 100 rows of 5 x 2 x 128256
    // 108.4 and 105.3 us a call; without one it is as fast one way, 256 rows of 9 x 2 x 256000 448.9 and 446.2, and slower the other,
    // 200 of 5 x 2 x 128256 136.2 and 139.5)
    if (PAIR && MASKED && pis == 0)
      a = logit_segment<DT, AL, PAIR, MASKED>(p, base, row_step, logit_weights(p, 0, thr), p.cT, v0, v1, ragged);
    else if (PAIR && MASKED)
      a = logit_segment<DT, AL, PAIR, MASKED>(p, base, row_step, logit_weights(p, 1, thr), p.cT, v0, v1, ragged);
    else
      a = logit_segment<DT, AL, PAIR, MASKED>(p, base, row_step, logit_weights(p, pis, thr), p.cT, v0, v1, ragged);
    put(0, pack_soft(a.q, thr));
    put(1, pack_soft(a.c, thr));
  } else {
    const ArgPart2 a = logit_arg_segment<DT, AL, PAIR, MASKED>(p, base, row_step, logit_weights(p, pis, thr), v0, v1, ragged);
    put(0, pack_arg(a.q, thr));
    put(1, pack_arg(a.c, thr));
  }
}

// PAIR, MASKED: logit level with exactly two models, and with a mask (kernels of their own: straight code for each).  Ensembles: PAIR
// is for long shares, which fetch a vector when the place of one before it is free; short ones fetch eight at a time.
template <int DT, int MODE, bool AL, bool PAIR, bool MASKED>
__global__ void __launch_bounds__(kStreamThreads, 1) cos_stream_kernel(const __grid_constant__ KParams p) {
  constexpr bool kEns = (MODE == kEnsembleSample || MODE == kEnsembleGreedy);
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  // Launched while the kernel before it in the stream drains (programmatic dependent launch): its blocks take their places
  // as that kernel's blocks leave and wait here until it is complete and its writes are visible.  (Without the launch
  // attribute, and behind a kernel that never signals, this is the ordinary order of a stream.)  Where the caller
  // promises that the inputs were complete earlier, a warp sweeps its first part first and waits only before it writes.
  bool waited = p.inputs_settled == 0;
  if (waited) asm volatile("griddepcontrol.wait;" ::: "memory");
  // The drawing launch reads the counter offset before it waits for this launch.  The promise does not cover an offset in device
  // memory, so there it may start only when every block of this launch is gone, and so has waited (each has a part to write).
  if (waited || p.off_dev == nullptr) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (w >= p.st_warps) return;
  const int slots = record_slots<MODE>(p);
  int share = w, i0 = 0, i1 = p.n;
  if (kEns && p.st_split) {
    const int row = w / p.st_split, unit = row / p.n;
    share = unit * p.st_split + w - row * p.st_split;
    i0 = row - unit * p.n;
    i1 = i0 + 1;
  }
  for (long long x = worker_lo(p, share), end = worker_lo(p, share + 1); x < end;) {
    const int r = line_div(x, p.st_nv, p.st_inv_nv);
    const int o0 = static_cast<int>(x - static_cast<long long>(r) * p.st_nv);
    const int o1 = end - x < p.st_nv - o0 ? o0 + static_cast<int>(end - x) : p.st_nv;
    x += o1 - o0;
    const int b = r / p.P, j = r - b * p.P;
    const char* base = reinterpret_cast<const char*>(p.logits) +
                       (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
    int pis = 0;
    float thr = -INFINITY;
    if (!kEns) {
      const int pi = proposer_of(p, b, j);
      pis = (pi >= 0 && pi < p.n) ? pi : 0;
      if (MASKED) thr = mask_bound(p, __ldcg(&p.mask_key[r]));
    }
    sweep_part<DT, MODE, AL, PAIR, MASKED>(p, base, o0, o1, i0, i1, pis, thr,
                                           p.st_rec + (static_cast<size_t>(r) + share) * slots, waited);
  }
}

// Forms of the streaming launch that decide while the sweep is under way.  One warp: the position (b, j) from its records `q`.
template <int DT, int MODE>
__device__ __forceinline__ void decide_and_publish(const KParams& p, Finish& fin, int b, int j, RecordRange q) {
  constexpr bool kEns = (MODE == kEnsembleSample || MODE == kEnsembleGreedy);
  constexpr bool kSample = (MODE == kEnsembleSample || MODE == kLogitSample);
  const int lane = threadIdx.x & 31, uidx = b * p.P + j, slots = record_slots<MODE>(p);
  const int g = slots <= 1 ? 32 : (slots <= 2 ? 16 : (slots <= 4 ? 8 : 4)), i = lane / g;
  const bool masked = !kEns && p.mask_model >= 0;
  const char* base = reinterpret_cast<const char*>(p.logits) +
                     (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
  const int pi = proposer_of(p, b, j);
  const bool pi_ok = (pi >= 0 && pi < p.n);
  const int pis = pi_ok ? pi : 0;
  const bool is_bonus = (j == p.gamma);
  const int draft = is_bonus ? 0 : __ldg(p.drafts + b * p.gamma + j);
  const bool draft_ok = is_bonus || (draft >= 0 && draft < p.V);
  const int at = is_bonus || !draft_ok ? -1 : draft;
  DraftLogit d = {0.0, 0.f};
  if (kSample && i < slots && lane % g == 0) d = draft_logit<DT, MODE>(p, base, i, pis, at);  // (asked for before the records are)
  const float thr = masked ? mask_bound(p, __ldcg(&p.mask_key[uidx])) : -INFINITY;
  if (i >= slots) q.count = 0;
  const Merged m = merge_slot<MODE, 8>(p, q, i, g, lane % g);
  if (i < slots && lane % g == 0) {
    if (kSample) {
      fin.fsoft[i] = m.soft;
      fin.pdraft[i] = draft_probability<MODE>(p, d, i, at, thr, m.soft, 1.0 / m.soft.s);
    } else {
      fin.farg[i] = m.arg;
    }
  }
  if (lane == 0) fin.thr = thr;
  __syncwarp();
  if (kSample && lane < slots) {  // kept for the drawing launch
    p.ustats[uidx].s[lane] = fin.fsoft[lane].s;
    p.ustats[uidx].ref[lane] = fin.fsoft[lane].ref;
  }
  if (kSample && lane == 31) p.ustats[uidx].thr32 = thr;
  if (lane == 0) {
    if (masked) p.mask_key[uidx] = 0u;  // ready for the next run
    unsigned rnd[4];
    philox4x32_10(static_cast<unsigned>(p.row_base + b), static_cast<unsigned>(j), offset_lo(p), offset_hi(p), p.seed_lo, p.seed_hi, rnd);
    decide_unit<DT, MODE>(p, fin, fin.dec, word_to_uniform(rnd[0]), word_to_uniform(rnd[1]), is_bonus, draft, draft_ok, pi, pi_ok, pis);
    const Decision& e = fin.dec;
    publish_unit(p, b, j, e.accept, e.status, e.cand, kSample ? e.drawable : __float_as_int(static_cast<float>(e.prob)), e.ratio, e.r_d,
                 e.q_d, e.S);
  }
  __syncwarp();
}

// For runs whose tokens the persistent kernel draws, which has no step that decides: the shares of the ordinary form, every part of a
// position reported (fence and counter); the warp that completes the position decides and publishes it.  Slower than deciding in
// the next launch (see above).
// PAIR: as in cos_stream_kernel.
template <int DT, int MODE, bool PAIR>
__global__ void __launch_bounds__(kStreamThreads, 1) cos_report_kernel(const __grid_constant__ KParams p) {
  constexpr bool kEns = (MODE == kEnsembleSample);
  __shared__ Finish fins[kStreamThreads / 32];
  const int lane = threadIdx.x & 31;
  const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (w >= p.st_workers) return;
  const int slots = record_slots<MODE>(p);
  bool waited = true;
  for (long long x = worker_lo(p, w), end = worker_lo(p, w + 1); x < end;) {
    const int r = line_div(x, p.st_nv, p.st_inv_nv);
    const int o0 = static_cast<int>(x - static_cast<long long>(r) * p.st_nv);
    const int o1 = end - x < p.st_nv - o0 ? o0 + static_cast<int>(end - x) : p.st_nv;
    x += o1 - o0;
    const int b = r / p.P, j = r - b * p.P;
    const char* base = reinterpret_cast<const char*>(p.logits) +
                       (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
    const int pi = kEns ? 0 : proposer_of(p, b, j);
    const int pis = (pi >= 0 && pi < p.n) ? pi : 0;
    sweep_part<DT, MODE, true, PAIR, false>(p, base, o0, o1, 0, p.n, pis, -INFINITY, p.st_rec + (static_cast<size_t>(r) + w) * slots, waited);
    const RecordRange q = records_of<MODE>(p, b, j);
    int prev = 0;
    if (lane == 0) {
      __threadfence();
      prev = atomicAdd(&p.st_arrivals[r], 1);
      __threadfence();
    }
    prev = __shfl_sync(0xffffffffu, prev, 0);
    if (prev != q.count - 1) continue;
    if (lane == 0) p.st_arrivals[r] = 0;  // ready for the next run
    decide_and_publish<DT, MODE>(p, fins[threadIdx.x >> 5], b, j, q);
  }
}

// For runs that leave positions unread behind a rejection their row has already reported.  A block takes a whole position at a time,
// the first positions of every row before the second ones, from a counter: 15 warps sweep it in equal contiguous parts, one
// decides and publishes the position before it and takes the next one while they do.  One barrier a position; two blocks on a
// multiprocessor, so that one streams while the other meets.
// What bounds it: how much is read before a row's rejection is known (592 positions are under way or next, in order), and memory latency
// and the barrier at what is read (1344 positions of 2 x 143360: half of the nominal DRAM rate, 4.2 and 2.4 warps waiting for them).  Shares of all warps over the first positions of every row, then over the second ones, and so on, read less (0.30
// of the positions instead of 0.48 for 256 rows of 256000 tokens), but the warps whose rows are rejected have nothing to do: whole calls
// 437 us sampled and 281 greedy, now 293 and 166.
__device__ __forceinline__ void early_barrier() {
  __syncwarp();
  asm volatile("barrier.sync 1, %0;" ::"n"(kEarlyThreads) : "memory");
}

template <int DT, int MODE, bool AL>
__global__ void __launch_bounds__(kEarlyThreads, kEarlyBlocks) cos_early_kernel(const __grid_constant__ KParams p) {
  constexpr bool kEns = (MODE == kEnsembleSample || MODE == kEnsembleGreedy);
  constexpr bool kSample = (MODE == kEnsembleSample || MODE == kLogitSample);
  __shared__ Finish fin;
  __shared__ int next[2];     // the position after the present one (by parity); num_units: none
  __shared__ int skipped[2];  // some warp left it unread
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool masked = !kEns && p.mask_model >= 0;
  const int slots = record_slots<MODE>(p);
  const int parts = (p.st_nv + p.st_share - 1) / p.st_share;
  int4* const recs = p.st_rec + static_cast<size_t>(blockIdx.x) * 2 * kEarlySweepers * slots;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if (threadIdx.x == 0) {
    next[0] = blockIdx.x;
    skipped[0] = skipped[1] = 0;
  }
  __syncthreads();
  // a position behind a rejection that its row has already published decides nothing (Sec. 3.1: the tokens after the first
  // rejection are discarded); it reports "not accepted, no candidate", which the row's scan never reaches, and has no
  // statistics (the log-sum-exps are exported from them)
  auto rejected = [&](int b, int j) {
    int rej = 0;
    if (lane == 0) rej = *reinterpret_cast<volatile int*>(&p.row_reject[b]);
    return __shfl_sync(0xffffffffu, rej, 0) < j;
  };
  auto leave = [&](int b, int j) {
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    if (lane < slots) p.ustats[b * p.P + j].s[lane] = nan;
    if (lane == 0) {
      if (masked) p.mask_key[b * p.P + j] = 0u;  // ready for the next run
      publish_unit(p, b, j, 0, 0, -1, kSample ? 0 : 0x7fc00000, nan, nan, nan, nan);
    }
    __syncwarp();
  };
  if (warp < kEarlySweepers) {
    bool waited = true;
#pragma unroll 1
    for (int k = 0;; k ^= 1) {
      const int unit = next[k];
      if (unit >= p.num_units) return;
      const int j = unit / p.B, b = unit - j * p.B;
      if (warp < parts) {
        if (rejected(b, j)) {  // (every warp looks for itself)
          if (lane == 0) skipped[k] = 1;
        } else {
          const int o0 = warp * p.st_share, o1 = o0 + p.st_share < p.st_nv ? o0 + p.st_share : p.st_nv;
          const char* base = reinterpret_cast<const char*>(p.logits) +
                             (static_cast<long long>(b) * p.s_row + static_cast<long long>(j) * p.s_pos) * Elem<DT>::bytes;
          const int pi = kEns ? 0 : proposer_of(p, b, j);
          const int pis = (pi >= 0 && pi < p.n) ? pi : 0;
          const float thr = masked ? mask_bound(p, __ldcg(&p.mask_key[b * p.P + j])) : -INFINITY;
          int4* rec = recs + (k * kEarlySweepers + warp) * slots;
          if (kEns || (p.n == 2 && !masked))
            sweep_part<DT, MODE, AL, true, false>(p, base, o0, o1, 0, p.n, pis, thr, rec, waited);
          else if (masked)
            sweep_part<DT, MODE, AL, false, true>(p, base, o0, o1, 0, p.n, pis, thr, rec, waited);
          else
            sweep_part<DT, MODE, AL, false, false>(p, base, o0, o1, 0, p.n, pis, thr, rec, waited);
        }
      }
      early_barrier();
    }
  }
#pragma unroll 1
  for (int k = 0;; k ^= 1) {
    const int unit = next[k];
    if (unit >= p.num_units) break;
    // the next position, while this one is swept
    int then = p.num_units;
#pragma unroll 1
    for (;;) {
      if (lane == 0) then = static_cast<int>(gridDim.x + atomicAdd(p.work_counter, 1u));
      then = __shfl_sync(0xffffffffu, then, 0);
      if (then >= p.num_units) break;
      const int tj = then / p.B, tb = then - tj * p.B;
      if (!rejected(tb, tj)) break;
      leave(tb, tj);
    }
    if (lane == 0) next[k ^ 1] = then;
    early_barrier();  // this position's records are written (and the warps go on with the next one)
    const int j = unit / p.B, b = unit - j * p.B;
    const bool skip = skipped[k] != 0;
    __syncwarp();
    if (skip) {
      if (lane == 0) skipped[k] = 0;
      leave(b, j);
    } else {
      decide_and_publish<DT, MODE>(p, fin, b, j, RecordRange{recs + k * kEarlySweepers * slots, parts});
    }
  }
  // the last block to leave puts the counters back, for the next run
  if (lane == 0 && atomicAdd(&p.work_counter[1], 1u) == gridDim.x - 1) p.work_counter[0] = p.work_counter[1] = 0u;
}

// Test hook, greedy runs: r is a handful of atoms.
template <int DT>
__global__ void cos_dump_atoms_kernel(const __grid_constant__ KParams p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int uidx = blockIdx.y;
  const UnitStats* st = &p.ustats[uidx];
  float* out = p.dump_r + static_cast<long long>(uidx) * p.V;
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < p.V; x += gridDim.x * blockDim.x) {
    float v = st->pad[0] < 0 ? __int_as_float(0x7fc00000) : 0.f;
    for (int k = 0; k < st->pad[0]; ++k)
      if (__float_as_int(st->ref[k]) == x) v = static_cast<float>(st->s[k]);
    out[x] = v;
  }
}

}  // namespace cosv

#endif  // COS_STREAM_CUH
