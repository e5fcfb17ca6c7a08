// CoS verification step for sm_100a: combine (Eq. 3-5), accept test (Eq. 6), residual / bonus sample and
// first-rejection scan (Sec. 3.1) for every row of a batch and every one of its gamma + 1 positions.
//
// A run is two launches (three for ensembles of one or of more than four models at T > 0), and one more in front of them for
// the plausibility mask:
//   mask       the plausibility threshold of every position (cos_stream.cuh);
//   streaming  stream the n logit rows of every (row, position) once from HBM: partial softmax statistics or argmaxes
//              (cos_stream.cuh);
//   drawing    merge them, take the accept tests in fp64, find every row's first rejection, write the row's outputs
//              (cos_decide.cuh; at T = 0 that is all), and draw the row's token: one more sweep of the one position that
//              needs it (cos_draw.cuh).
// Runs whose rows have their places on the device side by side, each on a cluster of blocks, are one launch that does all of it
// (cos_row.cuh, plan_row).
// Blocks wait for one another only at the hardware barrier of their cluster.
//
// This file is the host side of the library (contexts, launches, the C entry points).  The kernels are compiled in
// cos_bf16.cu, cos_f16.cu and cos_f32.cu (those of cos_row.cuh in cos_row_*.cu); cos_common.cuh holds constants, launch parameters, loads, Philox and softmax
// partials, cos_fused.cu the persistent one-launch kernel, cos_probe.cu the two streaming ceilings.

#include <mutex>
#include <type_traits>

#include "cos_common.cuh"
#include "cos_fused.h"
#include "cos_launch.h"

using namespace cosv;

namespace {

// ------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------
thread_local std::string g_create_error;

}  // namespace

struct cos_verify_ctx {
  cos_verify_config cfg;
  int sm_count;
  int clusters[kRowParts + 1];  // clusters of so many blocks that the device holds at once
  unsigned* d_work_counter;
  bool scratch_dirty;
  int4* d_st_rec;
  int* d_st_arrivals;
  unsigned* d_mask_key;
  // device scratch
  int* d_row_arrivals;
  int* d_row_reject;
  int4* d_unit_res;
  int* d_job_count;
  int2* d_jobs;
  UnitStats* d_ustats;
  int* d_row_draw;
  // optional per-stage timing (cos_verify_set_stage_timing)
  bool timing;
  cudaEvent_t ev[4];
  int ev_used;  // events recorded by the last run
  // optional staging for host-pointer runs
  // the one-launch form of a run (sampling modes the fused kernel covers, no cluster size requested)
  bool fused;      // the one-launch kernel covers this configuration (its scratch is allocated)
  bool use_fused;  // and runs take it (cos_verify_set_one_launch)
  bool draw_fused; // staged runs draw their tokens with that kernel's drawing items
  FusedPlan fplan;
  FusedScratch fscr;
  void* fused_mem[9];
  size_t fused_bytes[9];
  unsigned wait_limit;  // idle polls after which a block of the one-launch kernel gives up
  int test_drop;        // test hook: one streaming warp never reports its first item
  void* d_logits;
  int* h_small;   // host-pointer runs, pinned: drafts and proposers, then the outputs
  int* d_small;   // the same on the device
  std::string err;
};

namespace {

int mode_of(const cos_verify_config& c) {
  const bool greedy = (c.temperature == 0.0f);
  if (c.combine == COS_COMBINE_PROB_ENSEMBLE) return greedy ? kEnsembleGreedy : kEnsembleSample;
  return greedy ? kLogitGreedy : kLogitSample;
}

int entries_per_vec(int dtype) { return dtype == COS_DTYPE_F32 ? 4 : 8; }
int elem_bytes(int dtype) { return dtype == COS_DTYPE_F32 ? 4 : 2; }

bool fail(std::string* dst, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  *dst = buf;
  return false;
}

bool validate_config(const cos_verify_config& c, std::string* err) {
  if (c.n < 1 || c.n > COS_MAX_MODELS) return fail(err, "n = %d outside 1..%d", c.n, COS_MAX_MODELS);
  if (c.combine != COS_COMBINE_PROB_ENSEMBLE && c.combine != COS_COMBINE_LOGIT_LINEAR)
    return fail(err, "unknown combine %d", c.combine);
  if (c.dtype != COS_DTYPE_F32 && c.dtype != COS_DTYPE_BF16 && c.dtype != COS_DTYPE_F16)
    return fail(err, "unknown dtype %d", c.dtype);
  if (!(c.temperature >= 0.0f) || !isfinite(c.temperature)) return fail(err, "temperature must be finite and >= 0");
  if (c.gamma < 0) return fail(err, "gamma = %d must be >= 0", c.gamma);
  if (c.vocab < 1) return fail(err, "vocab = %d must be >= 1", c.vocab);
  if (c.max_batch < 1) return fail(err, "max_batch = %d must be >= 1", c.max_batch);
  if (static_cast<long long>(c.max_batch) * (c.gamma + 1) > 0x3fffffffLL) return fail(err, "max_batch * (gamma + 1) too large");
  double sum = 0.0;
  for (int i = 0; i < c.n; ++i) {
    if (!isfinite(c.weights[i])) return fail(err, "weight %d is not finite", i);
    sum += static_cast<double>(c.weights[i]);
  }
  if (c.combine == COS_COMBINE_PROB_ENSEMBLE) {
    for (int i = 0; i < c.n; ++i)
      if (c.weights[i] < 0.0f) return fail(err, "ensemble weight %d is negative", i);
    if (fabs(sum - 1.0) > 1e-6) return fail(err, "ensemble weights sum to %.9g, not 1", sum);
    if (c.mask_model >= 0) return fail(err, "the plausibility mask needs the logit-level combine");
  } else if (c.mask_model >= 0) {
    if (c.mask_model >= c.n) return fail(err, "mask_model = %d outside 0..n-1", c.mask_model);
    if (!(c.mask_alpha > 0.0f && c.mask_alpha <= 1.0f)) return fail(err, "mask_alpha must lie in (0, 1]");
  }
  if (c.mask_model < -1) return fail(err, "mask_model must be -1 or a model index");
  const int cs = c.cluster_size;
  if (!(cs == 0 || cs == 1 || cs == 2 || cs == 4 || cs == 8 || cs == 16))
    return fail(err, "cluster_size must be 0, 1, 2, 4, 8 or 16");
  return true;
}

// Channels of the drawing launch: two describe every mass at logit level (proposer and combined logits) and for up to
// two models; a channel per model otherwise.
int draw_channels(const cos_verify_config& c) {
  if (c.combine != COS_COMBINE_PROB_ENSEMBLE || c.n <= 2) return 2;
  return c.n <= 4 ? 4 : 8;
}

// Ensembles of one or of more than four models decide in a launch of their own.
bool decides_first(const cos_verify_config& c) { return c.combine == COS_COMBINE_PROB_ENSEMBLE && (c.n == 1 || c.n > 4); }

// How the drawing launch shares a position out.  The device holds 32 warps per multiprocessor (two channels) or 16; a
// position gets a cluster of blocks of 16, 8 or 4 warps, whichever leaves least of the device idle.  Clusters of more than four
// blocks are taken only where they need no more than two thirds of the device: they do not pack (32 clusters of 8 blocks
// of 16 warps, on paper a fit, run in two waves: 31.8 us a call instead of 25.2 for 32 rows of 32000 tokens; 64 of 8 blocks of 8
// warps 91 instead of 83 for 64 rows of 151936).  Fewer and smaller clusters: one row of 151936 tokens 18.5 us with 8 blocks of 16
// warps, 20.7 with 4, 25.2 with 2.
// A warp has a few chunks (one record of sums each), of eight steps where there is room for the records, so that the token is
// searched in few steps.
struct DrawPlan {
  int threads, parts, cs, chunks;
};
DrawPlan draw_plan(const cos_verify_config& c, long long units, int sm_count) {
  DrawPlan d;
  const int nsteps = (c.vocab + 32 * entries_per_vec(c.dtype) - 1) / (32 * entries_per_vec(c.dtype));
  const int ch = draw_channels(c), most = ch == 2 ? 32 : 16;
  int best = 0;
  for (int nw = ch == 8 ? 8 : 16; nw >= 4; nw /= 2) {
    const long long blocks = static_cast<long long>(sm_count) * (most / nw);
    long long parts = blocks / units;
    if (parts > 4) {
      const long long loose = blocks * 2 / 3 / units;
      parts = loose < 4 ? 4 : (loose > 8 ? 8 : loose);
    }
    if (parts > (nsteps + nw - 1) / nw) parts = (nsteps + nw - 1) / nw;
    if (parts < 1 && nw == 4) parts = 1;
    if (parts * nw > best) {
      best = static_cast<int>(parts) * nw;
      d.threads = nw * 32;
      d.parts = static_cast<int>(parts);
    }
  }
  const int mine = (nsteps + best - 1) / best, room = 768 / ch / best;  // steps and records of a warp
  d.chunks = (mine + 7) / 8 < room ? (mine + 7) / 8 : room;
  d.cs = (mine + d.chunks - 1) / d.chunks;
  return d;
}

// Threads of a block of the streaming launch: 1024 where the launch fills the device (of two blocks of 512 on a multiprocessor the
// older one's warps go first and leave it half empty in the end: 64 rows of 151936 tokens 86.0 us a call with two, 84.6 with one),
// 512 and 128 where it does not, so that it spreads over all of it.
constexpr int kStreamBlock = 512, kStreamFull = 1024, kStreamSmall = 128;

// Cut the line of `units` positions into shares for at most `workers` warps (see cos_stream.cuh).  Small runs take fewer warps, so
// that each has a few loads in flight, in small blocks, so that they spread over the device.  Where nine tenths of the warps are
// busy that way, every position is a whole number of shares (its end padded): a warp then has one part, not the end of one and
// the beginning of the next, one after the other (16 rows of 50001 tokens and three models: the last warp ended after 17 us, the
// average one after 10); and of an ensemble (`models` > 1) it has one model's, for the same reason.  Returns the block size.
int plan_line(KParams& p, const cos_verify_config& c, long long units, int models, long long workers, int sm_count) {
  const int E = entries_per_vec(c.dtype), nvec = c.vocab / E;
  int nv = p.vec_ok ? nvec : nvec - 2;  // (unaligned rows: the first vector and the last one go entry by entry)
  if (nv < 1) nv = 1;                   // nothing but ragged entries
  // at least four loads for each lane; eight (all still on their way at once) where that leaves most of the device idle anyway,
  // or for one model at a time: fewer records to merge
  // (with many vectors a warp the loads of one model after another leave no gap to speak of, and the split is coarser: 32 rows of 7
  // positions of 4 x 128256, 3030 vectors, 65 us in one, 68 apart; 24 rows of 5 of 4 x 48000, 608 vectors, 34.6 in one, 32.8 apart.
  // From 768 to 1200 or so apart was the faster one too: 4 x 80000, 1013 vectors, 48.1 in one, 41.8 apart, 2 x 80000 39.7 and 37.8)
  if (units * models * nv >= 768 * workers) models = 1;
  const long long rows = units * models;
  long long most = rows * nv / 128;
  if (most < 8LL * sm_count || models > 1) most /= 2;
  const bool small = workers > most;
  const long long busy = small ? (most < 1 ? 1 : most) : workers;
  long long each = busy / rows;  // shares of a row
  if (small && each < 1 && rows <= workers) each = 1;
  if (each >= 1 && (small || rows * each * 10 >= busy * 9)) {
    p.st_share = static_cast<int>(((nv + each - 1) / each + 7) / 8 * 8);
    p.st_nv = (nv + p.st_share - 1) / p.st_share * p.st_share;
    p.st_line = units * p.st_nv;
    p.st_split = models > 1 ? p.st_nv / p.st_share : 0;
  } else {
    const long long line = units * nv;
    const long long shares = busy < line / 128 ? busy : (line / 128 < 1 ? 1 : line / 128);
    p.st_nv = nv;
    p.st_line = line;
    p.st_share = static_cast<int>(((line + shares - 1) / shares + 7) / 8 * 8);
    p.st_split = 0;
  }
  p.st_workers = static_cast<int>((p.st_line + p.st_share - 1) / p.st_share);
  p.st_warps = p.st_split ? p.st_workers * models : p.st_workers;
  p.st_inv_nv = 1.0 / p.st_nv;
  p.st_inv_share = 1.0 / p.st_share;
  const int slots = c.combine == COS_COMBINE_PROB_ENSEMBLE ? c.n : 2;
  p.slot_inv = (65536 + slots - 1) / slots;
  return p.st_warps <= 16LL * sm_count ? kStreamSmall : (p.st_warps <= 28LL * sm_count ? kStreamBlock : kStreamFull);
}

// The streaming launch with early exit (cos_early_kernel): a block a position, st_workers blocks.
int plan_positions(KParams& p, const cos_verify_config& c, int sm_count) {
  const int nvec = c.vocab / entries_per_vec(c.dtype), nv = p.vec_ok ? nvec : nvec - 2;
  p.st_nv = nv < 1 ? 1 : nv;
  p.st_share = ((p.st_nv + kEarlySweepers - 1) / kEarlySweepers + 7) / 8 * 8;
  p.st_workers = p.num_units < kEarlyBlocks * sm_count ? p.num_units : kEarlyBlocks * sm_count;
  return kEarlyThreads;
}

// Whether the hint to leave positions unread is taken.  It needs the decisions while the sweep is under way (cos_early_kernel, a block a
// position), which costs 20 to 40 us more than the streaming launch and what follows it, and where a block has few
// positions all are under way before a rejection is known.  Whole calls without and with it, in us: 256 rows of 9 positions of 2 x 128256 bf16
// (1.2 GB) 221 and 195, 512 rows of 2 x 50001 (0.9 GB) 335 and 246, 128 rows of 3 x 128256 with a mask (0.9 GB) 284 and 251, but
// 128 rows of 2 x 128256 (0.6 GB) 122 and 136, 512 rows of 2 x 32000 (0.6 GB) 137 and 149, and 64 rows of 7 positions of 8 x 128256 (0.9 GB,
// one and a half positions a block) 233 and 303.
bool early_exit_pays(const cos_verify_config& c, long long units, int sm_count) {
  const long long blocks = static_cast<long long>(kEarlyBlocks) * sm_count;
  return units >= 3 * blocks && units * c.n * (c.vocab / entries_per_vec(c.dtype)) >= blocks * 160000;
}

// Warps of the streaming launch: what the device holds at once, or the cluster size's worth of blocks for every position.
long long stream_workers(const cos_verify_config& c, long long units, int sm_count) {
  const long long most = static_cast<long long>(sm_count) * 2 * (kStreamBlock / 32);
  const long long asked = units * c.cluster_size * (kStreamBlock / 32);
  return c.cluster_size > 0 && asked < most ? asked : most;
}

template <typename F>
cudaError_t by_dtype(int dtype, F f) {
  if (dtype == COS_DTYPE_F32) return f(std::integral_constant<int, COS_DTYPE_F32>());
  if (dtype == COS_DTYPE_BF16) return f(std::integral_constant<int, COS_DTYPE_BF16>());
  return f(std::integral_constant<int, COS_DTYPE_F16>());
}

// The streaming launch, before it the one that finds the plausibility thresholds, and after it, at T = 0, the one that
// decides (with early exit or a job list the streaming launch decides itself).
cudaError_t launch_stream(const cos_verify_config& c, int mode, KParams& p, long long workers, int sm_count, cudaStream_t stream) {
  return by_dtype(c.dtype, [&](auto dt) {
    constexpr int DT = decltype(dt)::value;
    cudaError_t e = cudaSuccess;
    if (p.mask_model >= 0) {
      const int threads = plan_line(p, c, p.num_units, 1, workers, sm_count);
      e = mask_launch<DT>(p, threads, stream);
    }
    const bool report = p.early_exit || p.use_jobs;
    const int apart = c.combine == COS_COMBINE_PROB_ENSEMBLE && !report ? c.n : 1;
    const int threads = p.early_exit ? plan_positions(p, c, sm_count) : plan_line(p, c, p.num_units, apart, workers, sm_count);
    if (e == cudaSuccess) e = stream_launch<DT>(p, mode, threads, stream);
    p.decide = report || decides_first(c) ? 0 : 1;
    const bool first = p.greedy || decides_first(c);
    if (e == cudaSuccess && !report && first) e = decide_launch<DT>(p, mode, stream);
    if (e == cudaSuccess && p.greedy && p.dump_r != nullptr) e = dump_launch<DT>(p, mode, stream);
    return e;
  });
}

// Runs of one launch: a cluster of blocks a row, all rows at once (cos_row.cuh).  Whether this one is, and its plan.  `clusters[k]`:
// clusters of k blocks that the device holds at once.
// A row has the largest clusters of which the device holds one for each row (16 blocks up to 7 rows, 6 for 16, 4 for 33, 2 for 48 on a B200).
// That leaves multiprocessors idle which the launches of whole batches use, so it pays where a block's part is small (`mine`: its vectors)
// or little is left idle (`spread`: vectors for each multiprocessor if all of them shared the work).  Device time in us of the launches
// apart and of this one (5 positions; models x vocabulary, bf16 where nothing is said; some 1300 calls of 1 to 148 rows, every type, were compared):
//   two models sampled: 1 row of 2 x 128256 15.6 and 15.8, of 6 x 2 x 151936 16.2 and 17.6, 7 of 2 x 32000 17.6 and 15.4, of 2 x 128256 24.1 and
//     17.7, 33 of 2 x 128256 39.0 and 35.9, 48 of 2 x 64000 32.2 and 36.1;
//   three and four: 1 row of 4 x 32000 16.3 and 18.2, 7 of 4 x 64000 24.1 and 21.3, 12 of them 26.1 and 31.2; with 50 positions shares of four models no
//     longer end where positions do, 7 rows of 4 x 4000 22.3 and 29.8;
//   logit level: 7 rows of 2 x 128256 26.8 and 18.6, with a mask 33.5 and 22.6, 48 of them 48.4 and 55.0, with a mask 62.2 and 71.2, 48 of
//     2 x 64000 35.7 and 34.7; 124 of 3 x 2 x 71936 with a mask 64.9 and 68.0; 16 of 3 x 64000 with a mask 40.1 and 36.5; 24 of 3 x 64000 33.8 and
//     35.1, 25 of 8 x 3 x 47488 fp16 39.3 and 44.0; 57 of 9 x 1 x 57664 fp16 41.5 and 44.1;
//   greedy (little to save but launches): 12 rows of 2 x 32000 7.4 and 7.7, 16 of them 8.8 and 7.7, 24 of 2 x 64000 12.1 and 13.1; logit
//     level: 4 rows of 2 x 64000 7.9 and 8.6, 7 of them 9.6 and 8.7, with a mask 14.9 and 11.6; 24 of 3 x 64000 20.0 and 25.8.
// Unaligned rows, whose vectors are cut out of two, keep a block busy for as long again (fp32 twice as long): two models of 50001, 16 rows 25.2 and 22.8, 24
// rows 27.2 and 28.7, fp32 12 rows 26.5 and 26.0, 16 rows 30.5 and 38.0; logit level 24 rows 29.5 and 27.7, 33 rows 34.5 and 36.2, with a mask in
// fp32 12 rows 35.0 and 32.4, 16 rows 37.6 and 49.7; greedy 16 rows 14.2 and 13.1, 24 rows 15.5 and 18.1.  With nothing idle it pays further (74 rows, two
// blocks each, 62.1 and 59.6; fp32 85.4 and 99.2).
// A position takes a warp its round trips, however few vectors it has, and a vocabulary of next to nothing leaves a few warps with all of them: one row of
// 500 positions of 2 x 7 at logit level 19 and 558, of 2 x 100 18.9 and 88.9; of two models of 1000 15.2 and 22.2.
bool plan_row(const cos_verify_config& c, const int* clusters, int sm_count, KParams& p) {
  const int mode = mode_of(c), ch = draw_channels(c);
  if (c.cluster_size > 0 || (mode == kEnsembleSample && (c.n < 2 || c.n > 4))) return false;
  int parts = 0;
  for (int k = 1; k <= kRowParts; ++k)
    if (clusters[k] >= p.B) parts = k;
  if (parts == 0 || p.B * parts > sm_count) return false;
  const long long pairs = static_cast<long long>(c.n) * p.P, nv = c.vocab / entries_per_vec(c.dtype);
  const long long mine = pairs * (nv < 192 ? 192 : nv) / parts, spread = pairs * nv * p.B / sm_count, beyond = mine - spread * 17 / 20;
  const bool full = (mine - spread) * 16 <= spread;                // nothing idle
  const long long further = c.dtype != COS_DTYPE_F32 ? 47000 : 0;  // (unaligned rows)
  bool pays;
  switch (mode) {
    case kEnsembleSample:
      if (ch == 2)
        pays = p.vec_ok ? beyond <= 10000 : mine <= 12000 || (full && mine <= further);
      else
        pays = p.P <= 16 && spread >= 2500 && mine <= (p.vec_ok ? 10000 : 8000);
      break;
    case kLogitSample:
      if (!p.vec_ok)
        pays = mine <= (c.n > 2 ? 18000 : (spread <= 8000 ? 17000 : 14000)) || (full && mine <= further);
      else if (c.n == 2)
        pays = beyond <= (c.mask_model < 0 || parts >= 6 ? 18000 : 14000);
      else
        pays = beyond <= (c.n == 1 ? 9000 : (c.mask_model >= 0 || parts >= 6 || full ? 12000 : 7300));
      break;
    case kEnsembleGreedy:
      pays = spread >= 3500 && (p.vec_ok ? beyond <= 4500 : mine <= 8000);
      break;
    default:
      if (!p.vec_ok)
        pays = spread >= 1600 && mine <= 12000 && mine - 2 * spread <= 2500;
      else if (c.n <= 2)
        pays = spread >= 2500 && beyond <= 8000;
      else
        pays = mine - 2 * spread <= 500 && mine - spread * 3 / 5 <= (c.dtype != COS_DTYPE_F32 && spread <= 10000 ? 7500 : 6200);
  }
  if (!pays) return false;
  const int warps = parts * (kRowThreads / 32);
  plan_line(p, c, p.P, c.combine == COS_COMBINE_PROB_ENSEMBLE ? c.n : 1, warps, parts);
  if (p.P > 4 * p.st_workers) return false;
  p.st_row = p.st_workers;
  p.draw_parts = parts;
  const int steps = (p.nsteps + warps - 1) / warps, room = kRowSums / ch / warps;  // steps and records of a warp
  p.draw_chunks = (steps + 7) / 8 < room ? (steps + 7) / 8 : room;
  p.draw_cs = (steps + p.draw_chunks - 1) / p.draw_chunks;
  return true;
}

// What plan_row asks of a device, once for each (for runs without a context; a context keeps its own).
constexpr int kMaxDevices = 64;
struct DeviceShape {
  int sm_count, clusters[kRowParts + 1];
};
cudaError_t device_shape(int device, DeviceShape* out) {
  static DeviceShape shapes[kMaxDevices];
  static std::mutex guard;
  std::lock_guard<std::mutex> lock(guard);
  DeviceShape fresh = {};
  DeviceShape& d = device >= 0 && device < kMaxDevices ? shapes[device] : fresh;
  if (d.sm_count == 0) {
    for (int k = 1; k <= kRowParts; ++k) d.clusters[k] = row_clusters(k);
    const cudaError_t e = cudaDeviceGetAttribute(&d.sm_count, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) {
      d.sm_count = 0;
      return e;
    }
  }
  *out = d;
  return cudaSuccess;
}

// The launches that draw the tokens: of every position (`all`: test hook, residual masses) or of one per row.
cudaError_t launch_draw(const cos_verify_config& c, KParams& p, bool all, int sm_count, cudaStream_t stream) {
  const bool ens = c.combine == COS_COMBINE_PROB_ENSEMBLE;
  const int units = all ? p.num_units : p.B;
  const DrawPlan d = draw_plan(c, units, sm_count);
  p.draw_all = all ? 1 : 0;
  p.draw_parts = d.parts;
  p.draw_cs = d.cs;
  p.draw_chunks = d.chunks;
  return by_dtype(c.dtype, [&](auto dt) {
    constexpr int DT = decltype(dt)::value;
    cudaError_t e = draw_launch<DT>(p, ens, draw_channels(c), units, d.threads, stream);
    if (e == cudaSuccess && p.dump_r != nullptr) e = dump_launch<DT>(p, mode_of(c), stream);
    return e;
  });
}

cos_status cuda_fail(cos_verify_ctx* ctx, const char* what, cudaError_t e) {
  char buf[256];
  snprintf(buf, sizeof(buf), "%s: %s", what, cudaGetErrorString(e));
  if (ctx)
    ctx->err = buf;
  else
    g_create_error = buf;
  return COS_ERR_CUDA;
}

// What a launch needs from the configuration and the arguments of a run (everything but the scratch pointers).
void fill_params(const cos_verify_config& c, const cos_verify_args* a, KParams& p) {
  memset(&p, 0, sizeof(p));
  p.logits = a->logits;
  p.s_model = a->stride_model;
  p.s_row = a->stride_row;
  p.s_pos = a->stride_pos;
  p.drafts = a->draft_tokens;
  p.proposer = a->proposer;
  p.n = c.n;
  p.V = c.vocab;
  p.gamma = c.gamma;
  p.P = c.gamma + 1;
  p.B = a->batch;
  p.mask_model = (c.combine == COS_COMBINE_LOGIT_LINEAR) ? c.mask_model : -1;
  const int E = entries_per_vec(c.dtype);
  const int eb = elem_bytes(c.dtype);
  p.vec_ok = (reinterpret_cast<uintptr_t>(a->logits) % 16 == 0) && ((a->stride_model * eb) % 16 == 0) &&
             ((a->stride_row * eb) % 16 == 0) && ((a->stride_pos * eb) % 16 == 0);
  p.nsteps = (c.vocab + 32 * E - 1) / (32 * E);
  p.flags = a->flags;
  p.num_units = a->batch * (c.gamma + 1);
  for (int i = 0; i < COS_MAX_MODELS; ++i) {
    p.w[i] = (i < c.n) ? c.weights[i] : 0.f;
    p.w64[i] = static_cast<double>(p.w[i]);
  }
  if (c.temperature > 0.0f) {
    p.cT = static_cast<float>(1.4426950408889634 / static_cast<double>(c.temperature));
    p.cT64 = static_cast<double>(p.cT);
  }
  p.ln_alpha = (p.mask_model >= 0) ? log(static_cast<double>(c.mask_alpha)) : 0.0;
  p.seed_lo = static_cast<unsigned>(a->seed);
  p.seed_hi = static_cast<unsigned>(a->seed >> 32);
  p.off_lo = static_cast<unsigned>(a->offset);
  p.off_hi = static_cast<unsigned>(a->offset >> 32);
  p.off_dev = reinterpret_cast<const unsigned long long*>(a->offset_device);
  p.row_base = a->row_base;
  p.accept_count = a->accept_count;
  p.out_tokens = a->out_tokens;
  p.row_status = a->row_status;
  p.diag = a->diag;
  p.dump_r = a->dump_r;
  p.bonus_prob = a->bonus_prob;
  p.per_pos = (a->flags & COS_RUN_PROPOSER_PER_POSITION) ? 1 : 0;
  p.bonus_model = (a->flags & COS_RUN_BONUS_FROM_MODEL) ? a->bonus_model : -1;
  p.greedy = (c.temperature == 0.0f) ? 1 : 0;
}

cos_status init_scratch(cos_verify_ctx* ctx, cudaStream_t stream) {
  const size_t rows = static_cast<size_t>(ctx->cfg.max_batch);
  const size_t units = rows * (static_cast<size_t>(ctx->cfg.gamma) + 1);
  cudaError_t e = cudaMemsetAsync(ctx->d_work_counter, 0, 4 * sizeof(unsigned), stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_st_arrivals, 0, units * sizeof(int), stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_mask_key, 0, units * sizeof(unsigned), stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_row_arrivals, 0, rows * sizeof(int), stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_row_reject, 0x7f, rows * sizeof(int), stream);  // "none yet"
  if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_job_count, 0, 2 * sizeof(int), stream);
  if (ctx->fused) {
    // counters, row words, arrival counters and the queue start at zero; the rest is written before it is read
    static const int kClear[] = {0, 1, 2, 4, 5, 6};
    for (int k : kClear)
      if (e == cudaSuccess) e = cudaMemsetAsync(ctx->fused_mem[k], 0, ctx->fused_bytes[k], stream);
  }
  if (e != cudaSuccess) return cuda_fail(ctx, "scratch reset", e);
  ctx->scratch_dirty = false;
  return COS_OK;
}

}  // namespace

extern "C" cos_status cos_verify_create(const cos_verify_config* config, cos_verify_ctx** out) {
  if (!config || !out) {
    g_create_error = "null argument";
    return COS_ERR_INVALID_ARG;
  }
  *out = nullptr;
  if (!validate_config(*config, &g_create_error)) return COS_ERR_INVALID_ARG;
  cudaError_t e = cudaSetDevice(config->device);
  if (e != cudaSuccess) return cuda_fail(nullptr, "cudaSetDevice", e);
  cos_verify_ctx* ctx = new (std::nothrow) cos_verify_ctx();
  if (!ctx) {
    g_create_error = "out of host memory";
    return COS_ERR_NOMEM;
  }
  ctx->cfg = *config;
  cudaDeviceProp prop;
  e = cudaGetDeviceProperties(&prop, config->device);
  if (e != cudaSuccess) {
    delete ctx;
    return cuda_fail(nullptr, "cudaGetDeviceProperties", e);
  }
  ctx->sm_count = prop.multiProcessorCount;
  DeviceShape shape;
  e = device_shape(config->device, &shape);
  if (e != cudaSuccess) {
    delete ctx;
    return cuda_fail(nullptr, "cudaDeviceGetAttribute", e);
  }
  memcpy(ctx->clusters, shape.clusters, sizeof(shape.clusters));
  const size_t rows = static_cast<size_t>(config->max_batch), P = static_cast<size_t>(config->gamma) + 1;
  bool ok = true;
  ok = ok && cudaMalloc(&ctx->d_work_counter, 256) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_row_arrivals, rows * sizeof(int)) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_row_reject, rows * sizeof(int)) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_unit_res, rows * P * sizeof(int4)) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_job_count, 256) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_jobs, (rows * P + rows) * sizeof(int2)) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_ustats, rows * P * sizeof(UnitStats)) == cudaSuccess;
  {
    // records of a slot for each model (logit level: two) for every position of the line and for every warp; with early exit two
    // positions' worth for every block
    const size_t line = rows * P + static_cast<size_t>(ctx->sm_count) * 2 * (kStreamBlock / 32);
    const size_t apiece = static_cast<size_t>(ctx->sm_count) * kEarlyBlocks * 2 * kEarlySweepers;
    const size_t recs = (line > apiece ? line : apiece) * (config->combine == COS_COMBINE_PROB_ENSEMBLE ? config->n : 2);
    ok = ok && cudaMalloc(&ctx->d_st_rec, recs * sizeof(int4)) == cudaSuccess;
  }
  ok = ok && cudaMalloc(&ctx->d_st_arrivals, rows * P * sizeof(int)) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_mask_key, rows * P * sizeof(unsigned)) == cudaSuccess;
  ok = ok && cudaMalloc(&ctx->d_row_draw, rows * sizeof(int)) == cudaSuccess;
  ctx->wait_limit = 1u << 20;
  ctx->test_drop = 0;
  ctx->fused = false;
  ctx->draw_fused = false;
  if (ok && config->cluster_size == 0 &&
      fused_covers(config->dtype, mode_of(*config), config->n, config->vocab, config->gamma,
                   config->combine == COS_COMBINE_LOGIT_LINEAR ? config->mask_model : -1,
                   static_cast<long long>(rows) * static_cast<long long>(P))) {
    int per_sm = 0;
    e = fused_occupancy(config->dtype, mode_of(*config), config->n, &per_sm);
    if (e != cudaSuccess || per_sm < 1) {
      (void)cudaGetLastError();
    } else {
      ctx->fplan = fused_plan(config->dtype, mode_of(*config), config->n, config->vocab, config->gamma, config->max_batch,
                              ctx->sm_count, per_sm);
      fused_scratch_bytes(ctx->fplan, config->vocab, config->dtype, config->gamma, config->max_batch, ctx->fused_bytes);
      for (int k = 0; k < 9; ++k) ok = ok && cudaMalloc(&ctx->fused_mem[k], ctx->fused_bytes[k]) == cudaSuccess;
      if (ok) {
        ctx->fscr.ctr = static_cast<unsigned*>(ctx->fused_mem[0]);
        ctx->fscr.row_word = static_cast<unsigned long long*>(ctx->fused_mem[1]);
        ctx->fscr.unit_arrivals = static_cast<int*>(ctx->fused_mem[2]);
        ctx->fscr.chunk_part = static_cast<SoftPart*>(ctx->fused_mem[3]);
        ctx->fscr.dq = static_cast<int*>(ctx->fused_mem[4]);
        ctx->fscr.row_draw = static_cast<int*>(ctx->fused_mem[5]);
        ctx->fscr.draw_arrivals = static_cast<int*>(ctx->fused_mem[6]);
        ctx->fscr.dzpart = static_cast<double*>(ctx->fused_mem[7]);
        ctx->fscr.srec = static_cast<double*>(ctx->fused_mem[8]);
        ctx->fused = true;
      }
    }
  }
  if (ok && config->host_staging) {
    const size_t V = static_cast<size_t>(config->vocab);
    ok = ok && cudaMalloc(&ctx->d_logits, static_cast<size_t>(config->n) * rows * P * V * elem_bytes(config->dtype)) == cudaSuccess;
    const size_t small = rows * (2 * P + 3 + 5 * P) * sizeof(int);
    ok = ok && cudaMalloc(&ctx->d_small, small) == cudaSuccess && cudaMallocHost(&ctx->h_small, small) == cudaSuccess;
  }
  if (!ok) {
    (void)cudaGetLastError();
    cos_verify_destroy(ctx);
    g_create_error = "device allocation failed";
    return COS_ERR_NOMEM;
  }
  cos_status st = init_scratch(ctx, nullptr);
  if (st == COS_OK) {
    e = cudaDeviceSynchronize();
    if (e != cudaSuccess) st = cuda_fail(ctx, "cudaDeviceSynchronize", e);
  }
  if (st != COS_OK) {
    g_create_error = ctx->err;
    cos_verify_destroy(ctx);
    return st;
  }
  *out = ctx;
  return COS_OK;
}

namespace {
// the launches of one run; `lse_done`: the optional log-sum-exps are written by them (not those that decide in the streaming launch)
cos_status run_launches(cos_verify_ctx* ctx, const cos_verify_args* a, void* cuda_stream, bool* lse_done) {
  if (!ctx) return COS_ERR_INVALID_ARG;
  if (!a) {
    ctx->err = "null args";
    return COS_ERR_INVALID_ARG;
  }
  const cos_verify_config& c = ctx->cfg;
  auto bad = [&](const char* m) {
    ctx->err = m;
    return COS_ERR_INVALID_ARG;
  };
  if (a->batch < 1 || a->batch > c.max_batch) return bad("batch outside 1..max_batch");
  if (!a->logits || !a->proposer || !a->accept_count || !a->out_tokens || !a->row_status) return bad("null device pointer");
  if (c.gamma > 0 && !a->draft_tokens) return bad("draft_tokens is null although gamma > 0");
  if (a->stride_model < 0 || a->stride_row < 0 || a->stride_pos < 0) return bad("negative stride");
  if (a->flags & ~(COS_RUN_ALL_RESIDUALS | COS_RUN_PROPOSER_PER_POSITION | COS_RUN_BONUS_FROM_MODEL | COS_RUN_EARLY_EXIT |
                   COS_RUN_INPUTS_SETTLED)) return bad("unknown flag bits");
  if ((a->flags & COS_RUN_BONUS_FROM_MODEL) && (a->bonus_model < 0 || a->bonus_model >= c.n))
    return bad("bonus_model outside [0, n)");
  if (a->bonus_prob && reinterpret_cast<uintptr_t>(a->bonus_prob) % 4) {
    ctx->err = "bonus_prob is not 4-byte aligned";
    return COS_ERR_ALIGNMENT;
  }
  if (a->offset_device && reinterpret_cast<uintptr_t>(a->offset_device) % 8) {
    ctx->err = "offset_device is not 8-byte aligned";
    return COS_ERR_ALIGNMENT;
  }
  const int eb = elem_bytes(c.dtype);
  if (reinterpret_cast<uintptr_t>(a->logits) % eb) {
    ctx->err = "logits pointer not aligned to its element type";
    return COS_ERR_ALIGNMENT;
  }
  if (reinterpret_cast<uintptr_t>(a->proposer) % 4 || reinterpret_cast<uintptr_t>(a->accept_count) % 4 ||
      reinterpret_cast<uintptr_t>(a->out_tokens) % 4 || reinterpret_cast<uintptr_t>(a->row_status) % 4 ||
      (a->draft_tokens && reinterpret_cast<uintptr_t>(a->draft_tokens) % 4) ||
      (a->diag && reinterpret_cast<uintptr_t>(a->diag) % 4) || (a->dump_r && reinterpret_cast<uintptr_t>(a->dump_r) % 4)) {
    ctx->err = "an int32/float pointer is not 4-byte aligned";
    return COS_ERR_ALIGNMENT;
  }
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaSetDevice(c.device);
  if (e != cudaSuccess) return cuda_fail(ctx, "cudaSetDevice", e);
  if (ctx->scratch_dirty) {
    cos_status st = init_scratch(ctx, stream);
    if (st != COS_OK) return st;
  }

  KParams p;
  fill_params(c, a, p);
  p.work_counter = ctx->d_work_counter;
  p.row_arrivals = ctx->d_row_arrivals;
  p.row_reject = ctx->d_row_reject;
  p.early_exit = (a->flags & COS_RUN_EARLY_EXIT) ? 1 : 0;
  p.unit_res = ctx->d_unit_res;
  p.job_count = ctx->d_job_count;
  p.jobs = ctx->d_jobs;
  p.ustats = ctx->d_ustats;
  p.st_rec = ctx->d_st_rec;
  p.st_arrivals = ctx->d_st_arrivals;
  p.mask_key = ctx->d_mask_key;
  p.row_draw = ctx->d_row_draw;
  p.max_jobs = p.num_units + a->batch;

  const int mode = mode_of(c);
  const bool draws = (mode == kEnsembleSample || mode == kLogitSample);
  // One launch does the whole run where the fused kernel covers it: aligned rows, no test hook.  (The hint to
  // leave positions unread is not taken there: every position is read once.)
  if (ctx->fused && ctx->use_fused && p.vec_ok && a->dump_r == nullptr && !(a->flags & COS_RUN_ALL_RESIDUALS)) {
    p.early_exit = 0;
    ctx->scratch_dirty = true;
    if (ctx->timing) cudaEventRecord(ctx->ev[0], stream);
    e = fused_launch(c.dtype, mode, p, ctx->fplan, ctx->fscr, ctx->wait_limit, ctx->test_drop, false, stream);
    if (e != cudaSuccess) return cuda_fail(ctx, "kernel launch (one-launch form)", e);
    if (ctx->timing) cudaEventRecord(ctx->ev[1], stream);
    ctx->ev_used = 2;
    ctx->scratch_dirty = (ctx->test_drop != 0);  // a run that was made to give up leaves its counters behind
    return COS_OK;
  }
  ctx->scratch_dirty = true;  // cleared below once the launches are known to be queued
  if (ctx->timing) cudaEventRecord(ctx->ev[0], stream);
  const bool all = draws && ((a->dump_r != nullptr) || (a->flags & COS_RUN_ALL_RESIDUALS));
  // what it overlaps with is the end of the previous call's drawing launch, where one block per row goes on alone; a
  // drawing launch of more rows than the device has multiprocessors leaves nothing to fill (workload 5 was 12 us slower with
  // it), and greedy runs have no drawing launch
  p.inputs_settled = ((a->flags & COS_RUN_INPUTS_SETTLED) && draws && !all && !p.early_exit && p.mask_model < 0 &&
                      p.num_units >= ctx->sm_count && a->batch <= ctx->sm_count)
                         ? 1
                         : 0;
  const bool by_items = draws && !all && ctx->fused && ctx->draw_fused && p.vec_ok && a->lse == nullptr;
  p.use_jobs = by_items ? 1 : 0;
  const long long workers = stream_workers(c, p.num_units, ctx->sm_count);
  if (a->dump_r != nullptr || !early_exit_pays(c, p.num_units, ctx->sm_count)) p.early_exit = 0;
  if (!p.early_exit && !by_items && !all && a->dump_r == nullptr && plan_row(c, ctx->clusters, ctx->sm_count, p)) {
    p.lse = a->lse;
    *lse_done = p.lse != nullptr;
    e = by_dtype(c.dtype, [&](auto dt) { return row_launch<decltype(dt)::value>(p, mode, draw_channels(c), stream); });
    if (e != cudaSuccess) return cuda_fail(ctx, "kernel launch (rows at once)", e);
    if (ctx->timing) cudaEventRecord(ctx->ev[1], stream);
    ctx->ev_used = 2;
    ctx->scratch_dirty = false;
    return COS_OK;
  }
  const bool report = p.early_exit || by_items;
  p.lse = report ? nullptr : a->lse;
  *lse_done = p.lse != nullptr;
  p.keep_stats = (a->dump_r != nullptr || decides_first(c)) ? 1 : 0;
  e = launch_stream(c, mode, p, workers, ctx->sm_count, stream);
  if (e != cudaSuccess) return cuda_fail(ctx, "kernel launch (streaming)", e);
  if (ctx->timing) cudaEventRecord(ctx->ev[1], stream);
  ctx->ev_used = 2;
  if (draws) {
    if (by_items) {
      // the tokens are drawn by the persistent kernel's drawing items (any block takes any chunk of any row)
      e = fused_launch(c.dtype, mode, p, ctx->fplan, ctx->fscr, ctx->wait_limit, 0, true, stream);
      if (e != cudaSuccess) return cuda_fail(ctx, "kernel launch (drawing items)", e);
    } else {
      e = launch_draw(c, p, all, ctx->sm_count, stream);
      if (e != cudaSuccess) return cuda_fail(ctx, "kernel launch (drawing)", e);
    }
    if (ctx->timing) cudaEventRecord(ctx->ev[2], stream);
    ctx->ev_used = 3;
  }
  // (the kernels leave the scratch as they found it: every run starts from the same state with the same arguments)
  ctx->scratch_dirty = false;
  return COS_OK;
}

}  // namespace

namespace {
// The log-sum-exp behind every softmax of a position, from the merged statistics a run that decides in its first launch leaves
// per position.  One thread per (position, slot).
__global__ void export_lse_kernel(const UnitStats* ustats, const int4* unit_res, float* lse, int units, int slots, int sampling) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= units * slots) return;
  const int u = t / slots, k = t % slots;
  SoftPart f;
  f.s = ustats[u].s[k];
  f.ref = ustats[u].ref[k];
  lse[t] = log_sum_exp(f, sampling && !(__ldcg(&unit_res[u]).y & COS_ROW_NONFINITE));
}

}  // namespace

extern "C" cos_status cos_verify_run(cos_verify_ctx* ctx, const cos_verify_args* a, void* cuda_stream) {
  if (ctx && a && a->lse && reinterpret_cast<uintptr_t>(a->lse) % 4) {
    ctx->err = "lse is not 4-byte aligned";
    return COS_ERR_ALIGNMENT;
  }
  bool lse_done = false;
  const cos_status st = run_launches(ctx, a, cuda_stream, &lse_done);
  if (st != COS_OK || a->lse == nullptr || lse_done) return st;
  const cos_verify_config& c = ctx->cfg;
  const int units = a->batch * (c.gamma + 1);
  const int slots = (c.combine == COS_COMBINE_PROB_ENSEMBLE) ? c.n : 2;
  const int total = units * slots;
  export_lse_kernel<<<(total + 255) / 256, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(
      ctx->d_ustats, ctx->d_unit_res, a->lse, units, slots, c.temperature > 0.0f ? 1 : 0);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(ctx, "kernel launch (log-sum-exp export)", e);
  return COS_OK;
}

extern "C" cos_status cos_verify_run_host(cos_verify_ctx* ctx, const cos_verify_args* a, void* cuda_stream) {
  if (!ctx) return COS_ERR_INVALID_ARG;
  if (!a) {
    ctx->err = "null args";
    return COS_ERR_INVALID_ARG;
  }
  const cos_verify_config& c = ctx->cfg;
  if (!ctx->d_logits) {
    ctx->err = "context was created without host_staging";
    return COS_ERR_INVALID_ARG;
  }
  if (a->batch < 1 || a->batch > c.max_batch) {
    ctx->err = "batch outside 1..max_batch";
    return COS_ERR_INVALID_ARG;
  }
  if (a->dump_r || a->lse) {
    ctx->err = "dump_r and lse are not available for host-pointer runs";
    return COS_ERR_UNSUPPORTED;
  }
  if (!a->logits || !a->proposer || !a->accept_count || !a->out_tokens || !a->row_status || (c.gamma > 0 && !a->draft_tokens)) {
    ctx->err = "null host pointer";
    return COS_ERR_INVALID_ARG;
  }
  const long long V = c.vocab, P = c.gamma + 1, B = a->batch;
  if (a->stride_pos != V || a->stride_row != P * V || a->stride_model != B * P * V) {
    ctx->err = "host-pointer runs need contiguous [n][B][gamma+1][V] logits";
    return COS_ERR_INVALID_ARG;
  }
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaSetDevice(c.device);
  if (e != cudaSuccess) return cuda_fail(ctx, "cudaSetDevice", e);
  // The small arrays go by way of pinned memory of the context (the call waits for its launches, so that memory is free again when it
  // returns), which the kernels write directly: copies of their own, seven of them, were half of the call for one row.  The inputs
  // are copied together, but for one row of an ensemble, of which only the decisions read them (2 x 9 x 2000 bf16, in us, read where they are
  // and copied: one row 49.2 and 52.7, two 54.9 and 55.5, four 58.5 and 57.3, 64 rows 140.5 and 139.3).
  const size_t lbytes = static_cast<size_t>(c.n) * B * P * V * elem_bytes(c.dtype);
  const size_t ndraft = static_cast<size_t>(B * c.gamma), nprop = static_cast<size_t>((a->flags & COS_RUN_PROPOSER_PER_POSITION) ? B * P : B);
  int* out = ctx->h_small + ndraft + nprop;
  int* in = ctx->h_small;
  // the persistent kernel adds status bits with atomics, which are for device memory: its outputs are copied
  const bool items = ctx->fused && (ctx->use_fused || ctx->draw_fused);
  int* written = items ? ctx->d_small + ndraft + nprop : out;
  if (ndraft) memcpy(ctx->h_small, a->draft_tokens, ndraft * sizeof(int));
  memcpy(ctx->h_small + ndraft, a->proposer, nprop * sizeof(int));
  if (B > 1 || c.combine != COS_COMBINE_PROB_ENSEMBLE || items) {
    in = ctx->d_small;
    e = cudaMemcpyAsync(ctx->d_small, ctx->h_small, (ndraft + nprop) * sizeof(int), cudaMemcpyHostToDevice, stream);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(ctx->d_logits, a->logits, lbytes, cudaMemcpyHostToDevice, stream);
  if (e != cudaSuccess) {
    cudaStreamSynchronize(stream);
    return cuda_fail(ctx, "host to device copy", e);
  }
  cos_verify_args d = *a;
  d.flags &= ~COS_RUN_INPUTS_SETTLED;  // the inputs are what the copies above have just written
  d.logits = ctx->d_logits;
  d.draft_tokens = in;
  d.proposer = in + ndraft;
  d.accept_count = written;
  d.row_status = reinterpret_cast<unsigned*>(written + B);
  d.bonus_prob = a->bonus_prob ? reinterpret_cast<float*>(written + 2 * B) : nullptr;
  d.out_tokens = written + 3 * B;
  d.diag = a->diag ? reinterpret_cast<float*>(written + 3 * B + B * P) : nullptr;
  if (a->offset_device) {  // a host address here, like every other pointer of this call
    d.offset = *a->offset_device;
    d.offset_device = nullptr;
  }
  cos_status st = cos_verify_run(ctx, &d, stream);
  if (st != COS_OK) {
    cudaStreamSynchronize(stream);
    return st;
  }
  if (items) e = cudaMemcpyAsync(out, written, (3 * B + B * P * (a->diag ? 5 : 1)) * sizeof(int), cudaMemcpyDeviceToHost, stream);
  const cudaError_t waited = cudaStreamSynchronize(stream);
  if (e == cudaSuccess) e = waited;
  if (e != cudaSuccess) {
    ctx->scratch_dirty = true;
    return cuda_fail(ctx, "waiting for the launches", e);
  }
  memcpy(a->accept_count, out, B * sizeof(int));
  memcpy(a->row_status, out + B, B * sizeof(int));
  if (a->bonus_prob) memcpy(a->bonus_prob, out + 2 * B, B * sizeof(int));
  memcpy(a->out_tokens, out + 3 * B, B * P * sizeof(int));
  if (a->diag) memcpy(a->diag, out + 3 * B + B * P, B * P * 4 * sizeof(int));
  return COS_OK;
}

extern "C" cos_status cos_verify_set_stage_timing(cos_verify_ctx* ctx, int enable) {
  if (!ctx) return COS_ERR_INVALID_ARG;
  if (enable && !ctx->ev[0]) {
    for (int k = 0; k < 4; ++k) {
      cudaError_t e = cudaEventCreate(&ctx->ev[k]);
      if (e != cudaSuccess) return cuda_fail(ctx, "cudaEventCreate", e);
    }
  }
  ctx->timing = enable != 0;
  ctx->ev_used = 0;
  return COS_OK;
}

extern "C" cos_status cos_verify_get_stage_ms(cos_verify_ctx* ctx, float* ms, int32_t* count) {
  if (!ctx || !ms || !count) return COS_ERR_INVALID_ARG;
  *count = 0;
  if (!ctx->timing || ctx->ev_used < 2) {
    ctx->err = "no timed run to report";
    return COS_ERR_INVALID_ARG;
  }
  cudaError_t e = cudaEventSynchronize(ctx->ev[ctx->ev_used - 1]);
  for (int k = 0; e == cudaSuccess && k + 1 < ctx->ev_used; ++k) e = cudaEventElapsedTime(&ms[k], ctx->ev[k], ctx->ev[k + 1]);
  if (e != cudaSuccess) return cuda_fail(ctx, "stage timing", e);
  *count = ctx->ev_used - 1;
  return COS_OK;
}

extern "C" cos_status cos_verify_set_one_launch(cos_verify_ctx* ctx, int32_t enable) {
  if (!ctx) return COS_ERR_INVALID_ARG;
  if (enable && !ctx->fused) {
    ctx->err = "the one-launch form does not cover this configuration";
    return COS_ERR_UNSUPPORTED;
  }
  ctx->use_fused = (enable == 1);
  ctx->draw_fused = (enable == 2);
  return COS_OK;
}

extern "C" cos_status cos_verify_set_wait_limit(cos_verify_ctx* ctx, uint32_t polls, int32_t test_drop_report) {
  if (!ctx) return COS_ERR_INVALID_ARG;
  if (polls < 16) {
    ctx->err = "wait limit below 16 polls";
    return COS_ERR_INVALID_ARG;
  }
  ctx->wait_limit = polls;
  ctx->test_drop = test_drop_report ? 1 : 0;
  return COS_OK;
}

extern "C" cos_status cos_verify_get_info(const cos_verify_ctx* ctx, cos_verify_info* info) {
  if (!ctx || !info) return COS_ERR_INVALID_ARG;
  memset(info, 0, sizeof(*info));
  {
    // blocks of the streaming launch that share a position, and how many positions they share at once
    const long long units = static_cast<long long>(ctx->cfg.max_batch) * (ctx->cfg.gamma + 1);
    const long long blocks = stream_workers(ctx->cfg, units, ctx->sm_count) / (kStreamBlock / 32);
    const long long each = ctx->cfg.cluster_size > 0 ? ctx->cfg.cluster_size : (blocks + units - 1) / units;
    info->cluster_size = static_cast<int32_t>(each);
    info->max_clusters = static_cast<int32_t>((2LL * ctx->sm_count + each - 1) / each);
  }
  info->threads_per_block = kStreamBlock;
  info->sm_count = ctx->sm_count;
  {
    // ordinary runs (no test hook): the streaming launch and one that decides, or one or two that decide and draw; one
    // more for the mask
    const bool one_draw = !decides_first(ctx->cfg) || (ctx->fused && ctx->draw_fused);
    info->launches_per_run = (ctx->fused && ctx->use_fused) ? 1 : (ctx->cfg.temperature == 0.0f || one_draw ? 2 : 3);
    if (ctx->cfg.combine == COS_COMBINE_LOGIT_LINEAR && ctx->cfg.mask_model >= 0) ++info->launches_per_run;
  }
  info->reserved[0] = ctx->fused ? ctx->fplan.chunks : 1;
  info->reserved[1] = ctx->fused ? ctx->fplan.dchunks : 1;
  KParams p = {};
  p.B = ctx->cfg.max_batch;
  p.P = ctx->cfg.gamma + 1;
  p.vec_ok = 1;
  p.nsteps = (ctx->cfg.vocab + 32 * entries_per_vec(ctx->cfg.dtype) - 1) / (32 * entries_per_vec(ctx->cfg.dtype));
  const bool staged = !ctx->fused || !(ctx->use_fused || ctx->draw_fused);
  info->reserved[2] = ((ctx->fused && ctx->use_fused) ? 1 : 0) | ((ctx->fused && ctx->draw_fused) ? 2 : 0) |
                      (staged && plan_row(ctx->cfg, ctx->clusters, ctx->sm_count, p) ? 4 : 0);
  return COS_OK;
}

extern "C" cos_status cos_verify_destroy(cos_verify_ctx* ctx) {
  if (!ctx) return COS_OK;
  (void)cudaSetDevice(ctx->cfg.device);
  (void)cudaDeviceSynchronize();
  cudaFree(ctx->d_work_counter);
  cudaFree(ctx->d_row_arrivals);
  cudaFree(ctx->d_row_reject);
  cudaFree(ctx->d_job_count);
  cudaFree(ctx->d_jobs);
  cudaFree(ctx->d_ustats);
  cudaFree(ctx->d_st_rec);
  cudaFree(ctx->d_st_arrivals);
  cudaFree(ctx->d_mask_key);
  cudaFree(ctx->d_row_draw);
  for (int k = 0; k < 4; ++k)
    if (ctx->ev[k]) cudaEventDestroy(ctx->ev[k]);
  cudaFree(ctx->d_unit_res);
  for (int k = 0; k < 9; ++k) cudaFree(ctx->fused_mem[k]);
  cudaFree(ctx->d_logits);
  cudaFree(ctx->d_small);
  cudaFreeHost(ctx->h_small);
  (void)cudaGetLastError();
  delete ctx;
  return COS_OK;
}

extern "C" const char* cos_verify_last_error(const cos_verify_ctx* ctx) {
  return ctx ? ctx->err.c_str() : g_create_error.c_str();
}

// ------------------------------------------------------------------------------------
// verification without a context and without any device allocation
// ------------------------------------------------------------------------------------
namespace {

// Scratch of the context-free entry point.  It is part of the library image: every device
// that loads the library holds these COS_STATIC_SCRATCH_BYTES until the process exits.
// Layout: [0, 256) unused | mask keys | unit results | records of the streaming launch | unit
// statistics | drawing positions.
static __device__ __align__(256) unsigned char g_static_scratch[COS_STATIC_SCRATCH_BYTES];

constexpr int kStaticWorkers = 5120;  // warps of a streaming launch there is room for
constexpr int kStaticMaxDevices = 64;
// Device address of g_static_scratch per device.  In host code the symbol itself is only a
// stand-in, never an address a kernel may use, so the address is asked for once per device.
unsigned char* g_static_addr[kStaticMaxDevices];
bool g_static_ready[kStaticMaxDevices];
std::mutex g_static_mutex;  // first calls from several host threads look the address up once

cos_status static_fail(cos_status st, const char* msg) {
  g_create_error = msg;
  return st;
}

}  // namespace

extern "C" cos_status cos_verify_run_static(const cos_verify_config* config, const cos_verify_args* a,
                                            void* cuda_stream) {
  if (!config || !a) return static_fail(COS_ERR_INVALID_ARG, "null argument");
  cos_verify_config c = *config;
  c.max_batch = COS_STATIC_MAX_BATCH;  // the array, not the caller, bounds the batch here
  if (!validate_config(c, &g_create_error)) return COS_ERR_INVALID_ARG;
  if (a->batch < 1 || a->batch > COS_STATIC_MAX_BATCH)
    return static_fail(COS_ERR_INVALID_ARG, "batch exceeds COS_STATIC_MAX_BATCH (1024) of the built-in scratch");
  const long long units = static_cast<long long>(a->batch) * (c.gamma + 1);
  if (units > COS_STATIC_MAX_POSITIONS)
    return static_fail(COS_ERR_INVALID_ARG,
                       "batch * (gamma + 1) exceeds COS_STATIC_MAX_POSITIONS (8192) of the built-in scratch");
  if (c.device < 0 || c.device >= kStaticMaxDevices) return static_fail(COS_ERR_INVALID_ARG, "device ordinal out of range");
  if (!a->logits || !a->proposer || !a->accept_count || !a->out_tokens || !a->row_status)
    return static_fail(COS_ERR_INVALID_ARG, "null device pointer");
  if (c.gamma > 0 && !a->draft_tokens) return static_fail(COS_ERR_INVALID_ARG, "draft_tokens is null although gamma > 0");
  if (a->stride_model < 0 || a->stride_row < 0 || a->stride_pos < 0) return static_fail(COS_ERR_INVALID_ARG, "negative stride");
  if (a->flags & ~(COS_RUN_ALL_RESIDUALS | COS_RUN_PROPOSER_PER_POSITION | COS_RUN_BONUS_FROM_MODEL | COS_RUN_EARLY_EXIT |
                   COS_RUN_INPUTS_SETTLED)) return static_fail(COS_ERR_INVALID_ARG, "unknown flag bits");
  if ((a->flags & COS_RUN_BONUS_FROM_MODEL) && (a->bonus_model < 0 || a->bonus_model >= c.n))
    return static_fail(COS_ERR_INVALID_ARG, "bonus_model outside [0, n)");
  if (a->bonus_prob && reinterpret_cast<uintptr_t>(a->bonus_prob) % 4)
    return static_fail(COS_ERR_ALIGNMENT, "bonus_prob is not 4-byte aligned");
  if (a->offset_device && reinterpret_cast<uintptr_t>(a->offset_device) % 8)
    return static_fail(COS_ERR_ALIGNMENT, "offset_device is not 8-byte aligned");
  if (a->lse) return static_fail(COS_ERR_UNSUPPORTED, "lse is not available from the allocation-free entry point");
  const int eb = elem_bytes(c.dtype);
  if (reinterpret_cast<uintptr_t>(a->logits) % eb) return static_fail(COS_ERR_ALIGNMENT, "logits pointer not aligned to its element type");
  if (reinterpret_cast<uintptr_t>(a->proposer) % 4 || reinterpret_cast<uintptr_t>(a->accept_count) % 4 ||
      reinterpret_cast<uintptr_t>(a->out_tokens) % 4 || reinterpret_cast<uintptr_t>(a->row_status) % 4 ||
      (a->draft_tokens && reinterpret_cast<uintptr_t>(a->draft_tokens) % 4) ||
      (a->diag && reinterpret_cast<uintptr_t>(a->diag) % 4) || (a->dump_r && reinterpret_cast<uintptr_t>(a->dump_r) % 4))
    return static_fail(COS_ERR_ALIGNMENT, "an int32/float pointer is not 4-byte aligned");

  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  cudaError_t e = cudaSetDevice(c.device);
  if (e != cudaSuccess) return cuda_fail(nullptr, "cudaSetDevice", e);
  {
    std::lock_guard<std::mutex> guard(g_static_mutex);
    if (!g_static_ready[c.device]) {
      // once per device, with that device current: the device address of the built-in array
      void* addr = nullptr;
      e = cudaGetSymbolAddress(&addr, g_static_scratch);
      if (e != cudaSuccess || addr == nullptr) return cuda_fail(nullptr, "cudaGetSymbolAddress(built-in scratch)", e);
      g_static_addr[c.device] = static_cast<unsigned char*>(addr);
      g_static_ready[c.device] = true;
    }
  }
  DeviceShape shape;
  e = device_shape(c.device, &shape);
  if (e != cudaSuccess) return cuda_fail(nullptr, "cudaDeviceGetAttribute", e);
  const int sm_count = shape.sm_count;

  // carve the array; what must start clean comes first and is cleared on the caller's stream before the kernels
  const bool draws = c.temperature > 0.0f;
  const bool all = draws && ((a->dump_r != nullptr) || (a->flags & COS_RUN_ALL_RESIDUALS));
  const bool masked = c.combine == COS_COMBINE_LOGIT_LINEAR && c.mask_model >= 0;
  const size_t n_units = static_cast<size_t>(units);
  unsigned char* basep = g_static_addr[c.device];
  unsigned* d_mask_key = reinterpret_cast<unsigned*>(basep + 256);
  // (only the mask keys have to start clean: without a mask nothing in the array is read before the launches write it)
  if (masked) e = cudaMemsetAsync(d_mask_key, 0, n_units * sizeof(unsigned), stream);
  if (e != cudaSuccess) return cuda_fail(nullptr, "clearing the built-in scratch", e);
  int4* d_unit_res = reinterpret_cast<int4*>(basep + 256 + 4 * COS_STATIC_MAX_POSITIONS);
  int4* d_st_rec = d_unit_res + COS_STATIC_MAX_POSITIONS;
  UnitStats* d_ustats = reinterpret_cast<UnitStats*>(d_st_rec + COS_MAX_MODELS * (COS_STATIC_MAX_POSITIONS + kStaticWorkers));
  static_assert(sizeof(UnitStats) == 112, "COS_STATIC_SCRATCH_BYTES assumes 112 bytes of statistics per position");
  int* d_row_draw = reinterpret_cast<int*>(d_ustats + COS_STATIC_MAX_POSITIONS);

  KParams p;
  fill_params(c, a, p);
  p.num_units = static_cast<int>(units);
  // (the hint to leave positions unread is not taken here)
  p.early_exit = 0;
  p.unit_res = d_unit_res;
  p.ustats = d_ustats;
  p.st_rec = d_st_rec;
  p.mask_key = d_mask_key;
  p.row_draw = d_row_draw;

  if (!all && a->dump_r == nullptr && sm_count * (kRowThreads / 32) <= kStaticWorkers && plan_row(c, shape.clusters, sm_count, p)) {
    e = by_dtype(c.dtype, [&](auto dt) { return row_launch<decltype(dt)::value>(p, mode_of(c), draw_channels(c), stream); });
    if (e != cudaSuccess) return cuda_fail(nullptr, "kernel launch (rows at once)", e);
    return COS_OK;
  }
  long long workers = stream_workers(c, units, sm_count);
  if (workers > kStaticWorkers) workers = kStaticWorkers;
  p.keep_stats = (a->dump_r != nullptr || decides_first(c)) ? 1 : 0;
  e = launch_stream(c, mode_of(c), p, workers, sm_count, stream);
  if (e != cudaSuccess) return cuda_fail(nullptr, "kernel launch (streaming)", e);
  if (draws) {
    e = launch_draw(c, p, all, sm_count, stream);
    if (e != cudaSuccess) return cuda_fail(nullptr, "kernel launch (drawing)", e);
  }
  return COS_OK;
}
