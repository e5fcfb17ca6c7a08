// Shared device helpers of the CoS verification kernels: element types, streaming loads, Philox4x32-10,
// the base-2 softmax accumulators and their reductions, and the launch parameters.
#ifndef COS_COMMON_CUH
#define COS_COMMON_CUH
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <string>

#include "cos_verify.h"

namespace cg = cooperative_groups;

namespace cosv {

constexpr int kNoReject = 0x7fffffff;
constexpr int kPackedP = 13;  // rows of up to this many positions keep their accept flags in the arrival word
constexpr int kDrawResidual = 0, kDrawR = 1, kDrawQ = 2;  // what a token is drawn from: max(0, r - q), r, or q
// The streaming launch with early exit: a block's threads, the warps of it that sweep, blocks on a multiprocessor.
constexpr int kEarlyThreads = 512, kEarlySweepers = kEarlyThreads / 32 - 1, kEarlyBlocks = 2;
constexpr double kBigShare = 1.0 / 256.0;  // probabilities above 2^-8 get fp64 treatment when tokens are drawn

enum Mode { kEnsembleSample = 0, kLogitSample = 1, kEnsembleGreedy = 2, kLogitGreedy = 3 };

struct UnitStats {  // what the drawing launch needs to know about one (row, position)
  double s[COS_MAX_MODELS];   // normalisers sum 2^(arg - ref)
  float ref[COS_MAX_MODELS];  // reference exponents
  float thr32;                // plausibility threshold
  int pad[3];
};

struct KParams {
  const void* logits;
  long long s_model, s_row, s_pos;  // element strides
  const int* drafts;
  const int* proposer;
  int n, V, gamma, P, B;
  int mask_model;
  int vec_ok;   // every row start is 16-byte aligned
  int nsteps;   // ceil(V / (32 * E))
  int flags;
  int num_units;
  int per_pos;      // proposer is [B][gamma+1] (the model that proposed each draft) instead of [B]
  int early_exit;   // positions after a row's known first rejection may be left unread
  int greedy;       // T = 0: nothing is drawn; the fourth word of a unit's result carries the bonus probability
  int bonus_model;  // >= 0: the token after gamma acceptances follows this model's own distribution; -1: the combined one
  int inputs_settled;  // the inputs may be read before the kernel ahead in the stream is complete
  int max_jobs;  // capacity of the job list
  float w[COS_MAX_MODELS];
  double w64[COS_MAX_MODELS];
  float cT;       // log2(e) / T in fp32 (T > 0)
  double cT64;    // the same value widened: the decision uses the constant the sweeps used
  double ln_alpha;
  unsigned seed_lo, seed_hi, off_lo, off_hi;
  const unsigned long long* off_dev;  // when set, the counter offset is read from device memory instead
  long long row_base;
  int* accept_count;
  int* out_tokens;
  unsigned* row_status;
  float* diag;
  float* dump_r;
  float* bonus_prob;
  // scratch owned by the context
  unsigned* work_counter;  // next position to be taken, blocks that have left (early exit); zero between runs
  int* row_arrivals;       // [B], zero between runs
  int* row_reject;         // [B]: earliest rejected position published so far; kNoReject between runs
  int4* unit_res;          // [B*P]: x = accept flag, y = status bits, z = candidate token, w = a token can be drawn
  int* job_count;          // length of the job list (persistent kernel, which also clears it)
  int2* jobs;              // x = b * P + j of a unit that draws a token (y unused)
  UnitStats* ustats;       // [B*P]: merged statistics, where a later launch reads them
  int use_jobs;            // the list of drawing positions is kept too (tokens drawn by the persistent kernel)
  // the streaming launch: a line of st_line vectors (st_nv for each position) in st_workers shares of st_share vectors (the last may
  // be shorter)
  int st_workers, st_nv, st_share;
  int st_split;            // ensembles: shares of a position, each model's a warp of its own; 0: a warp sweeps all models of its share
  int st_warps;            // warps of the launch
  int st_row;              // > 0: every row is a line of its own, in this many shares (st_workers, st_warps and st_line are a row's, too)
  long long st_line;
  double st_inv_nv, st_inv_share;  // one over them, for divisions
  int slot_inv;            // 65536 over the records of a (share, position) pair, rounded up: likewise
  int4* st_rec;            // records: statistics of a share's part of a position
  int* st_arrivals;        // [B*P]: warps that have reported; zero between runs
  unsigned* mask_key;      // [B*P]: largest logit of the gating model as an ordered integer; zero between runs
  // the drawing launch
  int* row_draw;           // [B]: the position of the row that draws its token, or -1
  int draw_all;            // it visits every position (test hook, residual masses)
  int decide;              // it also merges the records of the streaming launch and decides (else that is done)
  int keep_stats;          // ustats, unit_res and row_draw are wanted afterwards
  float* lse;              // [B*P][records of a pair]: the log-sum-exps go here from the launch that decides
  int draw_parts;          // blocks of a position's cluster
  int draw_cs, draw_chunks;  // steps of a chunk, chunks of a warp
};

// ------------------------------------------------------------------------------------
// small device helpers
// ------------------------------------------------------------------------------------
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ uint4 ldg_stream16(const void* p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

template <int DT>
struct Elem;
template <>
struct Elem<COS_DTYPE_F32> {
  static constexpr int E = 4;  // entries per 16-byte vector
  static constexpr int bytes = 4;
  static __device__ __forceinline__ void unpack(const uint4& r, float (&v)[4]) {
    v[0] = __uint_as_float(r.x);
    v[1] = __uint_as_float(r.y);
    v[2] = __uint_as_float(r.z);
    v[3] = __uint_as_float(r.w);
  }
  static __device__ __forceinline__ float load1(const void* row, long long x) {
    return __ldg(reinterpret_cast<const float*>(row) + x);
  }
};
template <>
struct Elem<COS_DTYPE_F16> {  // IEEE half: 8 entries per 16-byte vector, widened exactly
  static constexpr int E = 8;
  static constexpr int bytes = 2;
  static __device__ __forceinline__ void unpack(const uint4& r, float (&v)[8]) {
    const unsigned w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
      v[2 * k] = f.x;
      v[2 * k + 1] = f.y;
    }
  }
  static __device__ __forceinline__ float load1(const void* row, long long x) {
    return __half2float(__ldg(reinterpret_cast<const __half*>(row) + x));
  }
};
template <>
struct Elem<COS_DTYPE_BF16> {
  static constexpr int E = 8;
  static constexpr int bytes = 2;
  static __device__ __forceinline__ void unpack(const uint4& r, float (&v)[8]) {
    v[0] = __uint_as_float(r.x << 16);
    v[1] = __uint_as_float(r.x & 0xffff0000u);
    v[2] = __uint_as_float(r.y << 16);
    v[3] = __uint_as_float(r.y & 0xffff0000u);
    v[4] = __uint_as_float(r.z << 16);
    v[5] = __uint_as_float(r.z & 0xffff0000u);
    v[6] = __uint_as_float(r.w << 16);
    v[7] = __uint_as_float(r.w & 0xffff0000u);
  }
  static __device__ __forceinline__ float load1(const void* row, long long x) {
    unsigned short h = __ldg(reinterpret_cast<const unsigned short*>(row) + x);
    return __uint_as_float(static_cast<unsigned>(h) << 16);
  }
};

// One lane's chunk of a step: E consecutive entries starting at entry0.  Entries at or
// beyond V read as -inf (probability zero, never a maximum).
template <int DT>
__device__ __forceinline__ void load_chunk(const void* row, int entry0, int V, bool vec_ok,
                                           float (&v)[Elem<DT>::E]) {
  constexpr int E = Elem<DT>::E;
  if (vec_ok && entry0 + E <= V) {
    uint4 raw = ldg_stream16(reinterpret_cast<const char*>(row) + static_cast<long long>(entry0) * Elem<DT>::bytes);
    Elem<DT>::unpack(raw, v);
  } else {
#pragma unroll
    for (int k = 0; k < E; ++k) v[k] = (entry0 + k < V) ? Elem<DT>::load1(row, entry0 + k) : -INFINITY;
  }
}

// Philox4x32-10 (Salmon et al., SC'11): 10 rounds of two 32x32->64 multiplies and a
// Weyl key schedule.
__device__ __forceinline__ void philox4x32_10(unsigned c0, unsigned c1, unsigned c2, unsigned c3, unsigned k0,
                                              unsigned k1, unsigned (&out)[4]) {
#pragma unroll 1  // (a chain of latencies either way; ten copies of it are a kilobyte of instructions to fetch)
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    unsigned hi0 = __umulhi(0xD2511F53u, c0), lo0 = 0xD2511F53u * c0;
    unsigned hi1 = __umulhi(0xCD9E8D57u, c2), lo1 = 0xCD9E8D57u * c2;
    unsigned n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
  }
  out[0] = c0;
  out[1] = c1;
  out[2] = c2;
  out[3] = c3;
}

__device__ __forceinline__ double word_to_uniform(unsigned w) {
  return (2.0 * static_cast<double>(w >> 9) + 1.0) * 5.9604644775390625e-08;  // 2^-24
}

// Eq. 6: u <= min(1, r / q), 0 < u < 1, from the probabilities of the draft token (q = 0: the ratio is infinite, or 0 where r is 0 too).  Without the
// quotient, which costs the decisions 0.3 us (contrastive decoding of 8 rows of 32000 tokens 18.1 and 18.4 us).  Both sides are taken far from
// the subnormal numbers first: there the product rounds to 0, or up to r, and lets pass what the ratio rules out.
__device__ __forceinline__ bool accepts(double u, double r_d, double q_d) {
  const double up = 0x1p300;  // (probabilities: nothing overflows)
  return q_d > 0.0 ? u * (q_d * up) <= r_d * up : r_d > 0.0;
}

__device__ __forceinline__ double shfl_double(double x, int src) {
  int lo = __double2loint(x), hi = __double2hiint(x);
  lo = __shfl_sync(0xffffffffu, lo, src);
  hi = __shfl_sync(0xffffffffu, hi, src);
  return __hiloint2double(hi, lo);
}
__device__ __forceinline__ double shfl_up_double(double x, int d) {
  int lo = __double2loint(x), hi = __double2hiint(x);
  lo = __shfl_up_sync(0xffffffffu, lo, d);
  hi = __shfl_up_sync(0xffffffffu, hi, d);
  return __hiloint2double(hi, lo);
}

// ------------------------------------------------------------------------------------
// partial results exchanged lane -> warp -> block -> cluster
// ------------------------------------------------------------------------------------
struct SoftPart {  // sum over a set of tokens of 2^(arg - ref)
  double s;
  float ref;
  int pad;
};

// ln sum_x exp(l(x) / T) of merged statistics, NaN where there is none.
__device__ __forceinline__ float log_sum_exp(const SoftPart& f, bool there) {
  if (!there) return __int_as_float(0x7fc00000);
  return static_cast<float>((static_cast<double>(f.ref) + log2(f.s)) * 0.6931471805599453);
}
struct ArgPart {  // running maximum with the lowest index among equals
  double val;
  int idx;
  int bad;  // a NaN or +inf was seen
};

__device__ __forceinline__ bool arg_better(double v, int i, double bv, int bi) {
  return (v > bv) || (v == bv && i < bi);
}

// lane accumulator of a softmax normaliser in the base-2 domain: s = sum 2^(v*c - ref)
// Two fp32 operations in one instruction (sm_100 has packed forms of fma, add and mul: each half is the IEEE
// operation of its scalar twin, so results do not change; what is saved is an issue slot).
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, float b0, float b1, float c0, float c1) {
  asm("{\n.reg .b64 ra, rb, rc, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\nmov.b64 rc, {%6, %7};\n"
      "fma.rn.f32x2 rd, ra, rb, rc;\nmov.b64 {%0, %1}, rd;\n}\n"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void mul2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{\n.reg .b64 ra, rb, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\nmul.rn.f32x2 rd, ra, rb;\nmov.b64 {%0, %1}, rd;\n}\n"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}
__device__ __forceinline__ void add2(float& d0, float& d1, float a0, float a1, float b0, float b1) {
  asm("{\n.reg .b64 ra, rb, rd;\nmov.b64 ra, {%2, %3};\nmov.b64 rb, {%4, %5};\nadd.rn.f32x2 rd, ra, rb;\nmov.b64 {%0, %1}, rd;\n}\n"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b0), "f"(b1));
}

// The same on values that stay packed.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float lo2(f32x2 v) { return __uint_as_float(static_cast<unsigned>(v)); }
__device__ __forceinline__ float hi2(f32x2 v) { return __uint_as_float(static_cast<unsigned>(v >> 32)); }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ void add2_if(f32x2& acc, f32x2 v, float when_positive) {
  asm("{\n.reg .pred p;\nsetp.gt.f32 p, %2, 0f00000000;\n@p add.rn.f32x2 %0, %0, %1;\n}\n" : "+l"(acc) : "l"(v), "f"(when_positive));
}

// One entry of a 16-byte vector, and all of them in pairs of neighbours.
template <int DT>
__device__ __forceinline__ float entry(const uint4& r, int k) {
  const unsigned w[4] = {r.x, r.y, r.z, r.w};
  if (DT == COS_DTYPE_F32) return __uint_as_float(w[k & 3]);
  const unsigned h = w[(k >> 1) & 3];
  if (DT == COS_DTYPE_BF16) return __uint_as_float((k & 1) ? (h & 0xffff0000u) : (h << 16));
  const __half2 hh = *reinterpret_cast<const __half2*>(&h);
  return (k & 1) ? __high2float(hh) : __low2float(hh);
}
template <int DT>
__device__ __forceinline__ void unpack_pairs(const uint4& r, f32x2 (&x)[Elem<DT>::E / 2]) {
#pragma unroll
  for (int k = 0; k < Elem<DT>::E / 2; ++k) x[k] = pack2(entry<DT>(r, 2 * k), entry<DT>(r, 2 * k + 1));
}
template <int DT>
__device__ __forceinline__ uint4 neg_inf_vector() {
  const unsigned w = DT == COS_DTYPE_F32 ? 0xff800000u : (DT == COS_DTYPE_BF16 ? 0xff80ff80u : 0xfc00fc00u);
  return make_uint4(w, w, w, w);
}

// Entries [e0, e0 + E) of a row one by one; -inf beyond V.  Out of line: only the ends of a row come here.
template <int DT>
__device__ __noinline__ uint4 ragged_vector(const void* row, int e0, int V) {
  uint4 r = neg_inf_vector<DT>();
  if (DT == COS_DTYPE_F32) {
    const unsigned* src = reinterpret_cast<const unsigned*>(row);
    if (e0 < V) r.x = __ldg(src + e0);
    if (e0 + 1 < V) r.y = __ldg(src + e0 + 1);
    if (e0 + 2 < V) r.z = __ldg(src + e0 + 2);
    if (e0 + 3 < V) r.w = __ldg(src + e0 + 3);
    return r;
  }
  const unsigned short* src = reinterpret_cast<const unsigned short*>(row);
  unsigned short h[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) h[k] = (e0 + k < V) ? __ldg(src + e0 + k) : static_cast<unsigned short>(r.x & 0xffffu);
  return make_uint4(h[0] | (static_cast<unsigned>(h[1]) << 16), h[2] | (static_cast<unsigned>(h[3]) << 16),
                    h[4] | (static_cast<unsigned>(h[5]) << 16), h[6] | (static_cast<unsigned>(h[7]) << 16));
}

// Vectors of a row of V entries that can be fetched with aligned 16-byte loads staying inside the row: [lo, hi).
// AL: the rows are 16-byte aligned.  Otherwise a vector is cut out of two aligned neighbours, which leaves out the first
// one and the last entries.
struct VecRange {
  int lo, hi;
};
template <int DT, bool AL>
__device__ __forceinline__ VecRange whole_vectors(int V) {
  constexpr int E = Elem<DT>::E;
  VecRange r;
  r.lo = AL ? 0 : 1;
  r.hi = AL ? V / E : V / E - 1;
  return r;
}

// One of the whole vectors of a row.  An unaligned row (its offset from a 16-byte boundary is the same for every
// vector) costs two loads, the second one mostly a hit in L1, and a shift by whole words and by bits: about two
// instructions per entry more, where loads of single entries cost one load for each.
template <int DT, bool AL>
__device__ __forceinline__ uint4 load_whole(const char* row, int v) {
  if (AL) return ldg_stream16(row + static_cast<long long>(v) * 16);
  const unsigned off = static_cast<unsigned>(reinterpret_cast<unsigned long long>(row)) & 15u;
  const uint4* src = reinterpret_cast<const uint4*>(row - off) + v;
  const uint4 a = __ldg(src);
  if (off == 0u) return a;
  const uint4 b = __ldg(src + 1);
  unsigned w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  if (off & 8u) {
#pragma unroll
    for (int k = 0; k < 6; ++k) w[k] = w[k + 2];
  }
  if (off & 4u) {
#pragma unroll
    for (int k = 0; k < 5; ++k) w[k] = w[k + 1];
  }
  if (off & 2u) {
#pragma unroll
    for (int k = 0; k < 4; ++k) w[k] = __funnelshift_r(w[k], w[k + 1], 16);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}
// Any vector of a row; -inf beyond V.
template <int DT, bool AL>
__device__ __forceinline__ uint4 load_vector(const char* row, int v, int V, const VecRange& whole) {
  if (v >= whole.lo && v < whole.hi) return load_whole<DT, AL>(row, v);
  return ragged_vector<DT>(row, v * Elem<DT>::E, V);
}

// A lane's sum is measured against a fixed reference exponent, seeded from its first vector, so it is 1 at least.  Where that vector
// held nothing but -inf the reference is 0 until further notice, and a sum below this may have lost what it should hold
// to underflow (or is of nothing): such a lane goes through its vectors again with a running maximum, and one with nothing
// ends with the reference of an empty sum.
constexpr float kTinySum = 8.67361738e-19f;  // 2^-60

struct LaneSoft {
  float ref, s;
  // whether the fixed reference held (a lane without any vector is as `init` left it)
  __device__ __forceinline__ bool holds() const { return s < INFINITY && (s >= kTinySum || ref == -INFINITY); }
  __device__ __forceinline__ void init() {
    ref = -INFINITY;
    s = 0.f;
  }
  // reference exponent moves up with the running maximum (never overflows)
  template <int E>
  __device__ __forceinline__ void add_online(const float (&v)[E], float c) {
    float vmax = v[0];
#pragma unroll
    for (int k = 1; k < E; ++k) vmax = fmaxf(vmax, v[k]);
    float cand = vmax * c;
    if (cand > ref) {
      s *= ex2_approx(ref - cand);
      ref = cand;
    }
    float nref = (ref == -INFINITY) ? 0.f : -ref;
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < E; ++k) acc += ex2_approx(fmaf(v[k], c, nref));
    s += acc;
  }
  __device__ __forceinline__ void add_online1(float x, float c) {
    float cand = x * c;
    if (cand > ref) {
      s *= ex2_approx(ref - cand);
      ref = cand;
    }
    float nref = (ref == -INFINITY) ? 0.f : -ref;
    s += ex2_approx(fmaf(x, c, nref));
  }
  // reference exponent fixed (set from the first chunk); the caller asks whether it held
  template <int E>
  __device__ __forceinline__ void seed(const float (&v)[E], float c) {
    float vmax = v[0];
#pragma unroll
    for (int k = 1; k < E; ++k) vmax = fmaxf(vmax, v[k]);
    float cand = vmax * c;
    ref = (fabsf(cand) < INFINITY) ? floorf(cand) : 0.f;  // a whole number: sums with such references rescale exactly
    s = 0.f;
  }
  // the same with the packed forms of fma and add (same values, fewer instructions)
  template <int E>
  __device__ __forceinline__ void add_fixed2(const float (&v)[E], float c) {
    const float nref = -ref;
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int k = 0; k < E; k += 2) {
      float t0, t1;
      fma2(t0, t1, v[k], v[k + 1], c, c, nref, nref);
      add2(a0, a1, a0, a1, ex2_approx(t0), ex2_approx(t1));
    }
    s += a0 + a1;
  }
  template <int E>
  __device__ __forceinline__ void add_fixed(const float (&v)[E], float c) {
    const float nref = -ref;
    float a0 = 0.f, a1 = 0.f;
#pragma unroll
    for (int k = 0; k < E; k += 2) {
      a0 += ex2_approx(fmaf(v[k], c, nref));
      a1 += ex2_approx(fmaf(v[k + 1], c, nref));
    }
    s += a0 + a1;
  }
};

// sum of (ref, s) pairs held one per lane: common reference = the largest, fp64 sum
__device__ __forceinline__ SoftPart warp_reduce_soft(float ref, double s) {
  float R = ref;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, d));
  // references seeded by the sweep are whole numbers: the factor is then an exact power of two and cheap
  const float d = ref - R;
  double t;
  if (ref == R)
    t = s;
  else if (d == floorf(d) && d > -1000.f)
    t = s * __hiloint2double((1023 + static_cast<int>(d)) << 20, 0);
  else
    t = s * exp2(static_cast<double>(ref) - static_cast<double>(R));
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    int lo = __shfl_xor_sync(0xffffffffu, __double2loint(t), d);
    int hi = __shfl_xor_sync(0xffffffffu, __double2hiint(t), d);
    t += __hiloint2double(hi, lo);
  }
  SoftPart o;
  o.s = t;
  o.ref = R;
  o.pad = 0;
  return o;
}

// The sum of a warp's lanes and its reference exponent: the largest of theirs and 8, since the lanes together may hold more than 32
// bits do.  A lane's sum may reach 127 powers of two above its own reference, so the distance between references is taken in two steps
// (in one, a lane whose reference lay 127 below the largest was lost, whatever it held).
__device__ __forceinline__ float warp_sum_soft(const LaneSoft& a, float& R) {
  // lanes of one warp: fp32 is enough here, the errors of the 32 scale factors average out
  R = a.ref;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, d));
  const float far = fmaxf(a.ref - R, -300.f), half = floorf(0.5f * far);  // (an empty sum's reference is minus infinity)
  float t = a.s * ex2_approx(half - 4.f) * ex2_approx(far - half - 4.f);
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) t += __shfl_xor_sync(0xffffffffu, t, d);
  R += 8.f;
  return t;
}
__device__ __forceinline__ void warp_merge_soft(LaneSoft a, SoftPart* dst, int lane) {
  float R;
  const float t = warp_sum_soft(a, R);
  if (lane == 0) {
    dst->s = static_cast<double>(t);
    dst->ref = R;
  }
}

__device__ __forceinline__ ArgPart warp_reduce_arg(double val, int idx, int bad, int lane) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    double ov = shfl_double(val, lane ^ d);
    int oi = __shfl_xor_sync(0xffffffffu, idx, d);
    bad |= __shfl_xor_sync(0xffffffffu, bad, d);
    if (arg_better(ov, oi, val, idx)) {
      val = ov;
      idx = oi;
    }
  }
  ArgPart o;
  o.val = val;
  o.idx = idx;
  o.bad = bad;
  return o;
}

// The model whose distribution is q at position j of row b: the row's proposer, or the proposer of that draft
// when the caller gave one per position (Algorithm 2 verifies tokens of several proposers in one sequence).
// At the bonus position of a call that names a bonus model, q is that model's distribution: the token is
// then drawn from q (Sec. 3.3) by the machinery that otherwise draws from r.
__device__ __forceinline__ int proposer_of(const KParams& p, int b, int j) {
  if (j == p.gamma && p.bonus_model >= 0) return p.bonus_model;
  return p.proposer[p.per_pos ? b * p.P + j : b];
}

// Counter words 2 and 3 of the Philox call: from the arguments, or from device memory when the caller keeps
// the offset there (so that a captured graph can be replayed with fresh uniforms).
__device__ __forceinline__ unsigned offset_lo(const KParams& p) {
  return p.off_dev ? static_cast<unsigned>(__ldcg(p.off_dev)) : p.off_lo;
}
__device__ __forceinline__ unsigned offset_hi(const KParams& p) {
  return p.off_dev ? static_cast<unsigned>(__ldcg(p.off_dev) >> 32) : p.off_hi;
}

// ------------------------------------------------------------------------------------
// sweep 1: a block's slice of the vocabulary, threads interleaved over 16-byte vectors
// ------------------------------------------------------------------------------------
// Sweep 1 only forms sums, maxima and argmaxes, so any assignment of tokens to threads
// will do: each block reads its slice as consecutive 8 KB pieces (one vector per thread),
// which keeps the DRAM accesses of a block contiguous.
struct Slice {
  int v_lo, v_hi;  // whole 16-byte vectors [v_lo, v_hi) of the row (aligned layouts only)
  int e_lo, e_hi;  // single entries [e_lo, e_hi): the ragged tail, or everything when unaligned
};

// The channel arguments of one lane's vector at logit level: the proposer's entries and the combined logits (-inf outside
// the mask), packed in pairs of neighbouring tokens.  PAIR: exactly two models (straight code); MASKED: there is a plausibility
// mask.  `more(i)` fetches the vector of model i >= 2.
struct LogitWeights {
  float w0, w1;
  int pis, mask_model;
  float thr;
};
__device__ __forceinline__ uint4 pick_vector(bool first, const uint4& a, const uint4& b) {
  return make_uint4(first ? a.x : b.x, first ? a.y : b.y, first ? a.z : b.z, first ? a.w : b.w);
}
template <int DT, bool PAIR, bool MASKED, typename F>
__device__ __forceinline__ void logit_args(const KParams& p, const LogitWeights& lw, const uint4& r0, const uint4& r1, F more,
                                           f32x2 (&xq)[Elem<DT>::E / 2], f32x2 (&cmb)[Elem<DT>::E / 2]) {
  constexpr int H = Elem<DT>::E / 2;
  uint4 rq = pick_vector(lw.pis == 0, r0, r1), rm = MASKED ? pick_vector(lw.mask_model == 0, r0, r1) : rq;
  {
    f32x2 x[H];
    unpack_pairs<DT>(r0, x);
    const f32x2 w = pack2(lw.w0, lw.w0);
#pragma unroll
    for (int k = 0; k < H; ++k) cmb[k] = mul2(w, x[k]);
  }
  if (PAIR || p.n >= 2) {
    f32x2 x[H];
    unpack_pairs<DT>(r1, x);
    const f32x2 w = pack2(lw.w1, lw.w1);
#pragma unroll
    for (int k = 0; k < H; ++k) cmb[k] = fma2(w, x[k], cmb[k]);
  }
  if (!PAIR) {
    for (int i = 2; i < p.n; ++i) {
      const uint4 r = more(i);
      if (i == lw.pis) rq = r;
      if (i == lw.mask_model) rm = r;
      f32x2 x[H];
      unpack_pairs<DT>(r, x);
      const f32x2 w = pack2(p.w[i], p.w[i]);
#pragma unroll
      for (int k = 0; k < H; ++k) cmb[k] = fma2(w, x[k], cmb[k]);
    }
  }
  unpack_pairs<DT>(rq, xq);
  if (MASKED) {
    f32x2 x[H];
    unpack_pairs<DT>(rm, x);
#pragma unroll
    for (int k = 0; k < H; ++k)
      cmb[k] = pack2(lo2(x[k]) >= lw.thr ? lo2(cmb[k]) : -INFINITY, hi2(x[k]) >= lw.thr ? hi2(cmb[k]) : -INFINITY);
  }
}
__device__ __forceinline__ LogitWeights logit_weights(const KParams& p, int pis, float thr) {
  LogitWeights lw;
  lw.w0 = p.w[0];
  lw.w1 = p.w[1];
  lw.pis = pis;
  lw.mask_model = p.mask_model;
  lw.thr = thr;
  return lw;
}
__device__ __forceinline__ float pair_at(f32x2 v, int k) { return (k & 1) ? hi2(v) : lo2(v); }

// Softmax statistics of a logit-level combine over the slice `sl` of one (row, position): accq = the proposer's
// softmax, accc = the softmax of the combined logits sum_i w_i l_i (entries outside the plausibility mask count
// as -inf).  Fast form: fixed reference exponents seeded from the thread's first vector, one vector of every model
// per trip, the first two models fetched one trip ahead; overflow, underflow or a non-finite input falls back to the
// running-maximum form.  `tid` in [0, NT): the threads that share the slice.
template <int DT, int NT>
__device__ __forceinline__ void logit_soft_slice(const KParams& p, const char* base, const Slice& sl, int tid, int pis,
                                                 bool masked, float thr, LaneSoft& accq, LaneSoft& accc) {
  constexpr int E = Elem<DT>::E;
  auto row_of = [&](int i) -> const void* { return base + static_cast<long long>(i) * p.s_model * Elem<DT>::bytes; };
    const char* row0 = reinterpret_cast<const char*>(row_of(0));
    const long long row_step = p.s_model * Elem<DT>::bytes;
    // Fast form: fixed reference exponents seeded from the thread's first vector, one vector of every model
    // per trip, the first two models fetched one trip ahead (four loads in flight per thread).
    bool settled = false;
    {
      accq.init();
      accc.init();
      const bool pair = (p.n >= 2);
      uint4 nx0 = make_uint4(0u, 0u, 0u, 0u), nx1 = nx0;
      const int v0 = sl.v_lo + tid;
      if (v0 < sl.v_hi) {
        nx0 = ldg_stream16(row0 + static_cast<long long>(v0) * 16);
        if (pair) nx1 = ldg_stream16(row0 + row_step + static_cast<long long>(v0) * 16);
      }
      bool first = true;
      for (int v = v0; v < sl.v_hi; v += NT) {
        const uint4 a0 = nx0, a1 = nx1;
        {
          const int vn = v + NT;
          if (vn < sl.v_hi) {
            nx0 = ldg_stream16(row0 + static_cast<long long>(vn) * 16);
            if (pair) nx1 = ldg_stream16(row0 + row_step + static_cast<long long>(vn) * 16);
          }
        }
        float cmb[E], xq[E];
        unsigned inbits = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < E; ++k) cmb[k] = 0.f;
        auto take = [&](int i, const uint4& raw) {
          float x[E];
          Elem<DT>::unpack(raw, x);
          const float wi = p.w[i];
#pragma unroll
          for (int k = 0; k < E; k += 2) fma2(cmb[k], cmb[k + 1], wi, wi, x[k], x[k + 1], cmb[k], cmb[k + 1]);
          if (i == pis) {
#pragma unroll
            for (int k = 0; k < E; ++k) xq[k] = x[k];
          }
          if (masked && i == p.mask_model) {
            inbits = 0u;
#pragma unroll
            for (int k = 0; k < E; ++k) inbits |= (x[k] >= thr) ? (1u << k) : 0u;
          }
        };
        take(0, a0);
        if (pair) take(1, a1);
        for (int i = 2; i < p.n; ++i) take(i, ldg_stream16(row0 + i * row_step + static_cast<long long>(v) * 16));
        if (masked) {
#pragma unroll
          for (int k = 0; k < E; ++k) cmb[k] = (inbits & (1u << k)) ? cmb[k] : -INFINITY;
        }
        if (first) {
          accq.seed(xq, p.cT);
          accc.seed(cmb, p.cT);
          first = false;
        }
        accq.add_fixed2(xq, p.cT);
        accc.add_fixed2(cmb, p.cT);
      }
      for (int e = sl.e_lo + tid; e < sl.e_hi; e += NT) {
        float cmb = 0.f, xq = -INFINITY, xe = 0.f;
        for (int i = 0; i < p.n; ++i) {
          float x = Elem<DT>::load1(row_of(i), e);
          cmb = fmaf(p.w[i], x, cmb);
          if (i == pis) xq = x;
          if (i == p.mask_model) xe = x;
        }
        if (masked && !(xe >= thr)) cmb = -INFINITY;
        accq.add_online1(xq, p.cT);
        accc.add_online1(cmb, p.cT);
      }
      settled = accq.holds() && accc.holds();
    }
    // overflow, underflow or a non-finite input: the running-maximum form (two vectors of two models per trip)
    if (!settled) {
      accq.init();
      accc.init();
      // one model's vector: add to the combined logits; the proposer's row also feeds its own softmax,
      // the expert's row yields the mask bits
      auto take = [&](int i, const uint4& raw, float (&cmb)[E], unsigned& inbits) {
        float x[E];
        Elem<DT>::unpack(raw, x);
        const float wi = p.w[i];
#pragma unroll
        for (int k = 0; k < E; ++k) cmb[k] = fmaf(wi, x[k], cmb[k]);
        if (i == pis) {
          accq.add_online(x, p.cT);
        }
        if (masked && i == p.mask_model) {
          inbits = 0u;
#pragma unroll
          for (int k = 0; k < E; ++k) inbits |= (x[k] >= thr) ? (1u << k) : 0u;
        }
      };
      auto finish = [&](float (&cmb)[E], unsigned inbits) {
        if (masked) {
#pragma unroll
          for (int k = 0; k < E; ++k) cmb[k] = (inbits & (1u << k)) ? cmb[k] : -INFINITY;
        }
        accc.add_online(cmb, p.cT);
      };
      for (int v = sl.v_lo + tid; v < sl.v_hi; v += 2 * NT) {
        const bool have_b = (v + NT < sl.v_hi);
        const long long oa = static_cast<long long>(v) * 16;
        const long long ob = have_b ? oa + static_cast<long long>(NT) * 16 : oa;
        float ca[E], cb[E];
        unsigned ba = 0xffffffffu, bb = 0xffffffffu;
#pragma unroll
        for (int k = 0; k < E; ++k) ca[k] = cb[k] = 0.f;
        int i = 0;
        for (; i + 1 < p.n; i += 2) {  // two models, two vectors: four loads in flight
          const char* r0 = row0 + i * row_step;
          const char* r1 = r0 + row_step;
          const uint4 a0 = ldg_stream16(r0 + oa), b0 = ldg_stream16(r0 + ob);
          const uint4 a1 = ldg_stream16(r1 + oa), b1 = ldg_stream16(r1 + ob);
          take(i, a0, ca, ba);
          take(i + 1, a1, ca, ba);
          if (have_b) {
            take(i, b0, cb, bb);
            take(i + 1, b1, cb, bb);
          }
        }
        if (i < p.n) {
          const char* r0 = row0 + i * row_step;
          const uint4 a0 = ldg_stream16(r0 + oa), b0 = ldg_stream16(r0 + ob);
          take(i, a0, ca, ba);
          if (have_b) take(i, b0, cb, bb);
        }
        finish(ca, ba);
        if (have_b) finish(cb, bb);
      }
      for (int e = sl.e_lo + tid; e < sl.e_hi; e += NT) {
        float cmb = 0.f, xq = -INFINITY, xe = 0.f;
        for (int i = 0; i < p.n; ++i) {
          float x = Elem<DT>::load1(row_of(i), e);
          cmb = fmaf(p.w[i], x, cmb);
          if (i == pis) xq = x;
          if (i == p.mask_model) xe = x;
        }
        if (masked && !(xe >= thr)) cmb = -INFINITY;
        accq.add_online1(xq, p.cT);
        accc.add_online1(cmb, p.cT);
      }
    }
}

}  // namespace cosv

#endif  // COS_COMMON_CUH
