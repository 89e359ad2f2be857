// C ABI of the RCP W2A4 library: argument validation, launch configuration, status codes.
#include "../../include/rcp.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <utility>

#include "common.cuh"
#include "gemv_simple.cuh"
#include "gemv_stream.cuh"
#include "gemv_umma.cuh"
#include "gemv_w3.cuh"
#include "ldp_export.cuh"
#include "split_act16.cuh"
#include "pack.cuh"
#include "quantize_act.cuh"

namespace {

thread_local int g_last_cuda_error = 0;

int cuda_fail(cudaError_t e) {
  g_last_cuda_error = (int)e;
  return RCP_ERR_CUDA;
}

#define RCP_CUDA(call)                            \
  do {                                            \
    cudaError_t e__ = (call);                     \
    if (e__ != cudaSuccess) return cuda_fail(e__); \
  } while (0)

// Launches with programmatic stream serialization: the kernel may start while the preceding
// kernel on the stream is still running and must execute griddepcontrol.wait before it touches
// anything that kernel may read or write.
template <typename... KArgs, typename... Args>
cudaError_t launch_overlapped(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool k_ok(int K) { return K >= 64 && K <= rcp::kMaxK && K % 64 == 0; }

// Set by pack_weights_kernel when it meets a code above 3. One slot per call in flight (calls from several host
// threads or on several streams take different slots, so that none clears or reads another's flag).
constexpr unsigned kPackSlots = 64;
__device__ int g_pack_bad[kPackSlots];
std::atomic<unsigned> g_pack_next{0};

// ---------------------------------------------------------------------------------------------
// Streaming GEMV: launch plan.
struct StreamPlan {
  int nchunk, nchunk_total, nsplit, nphase, stages, grid;   // nchunk: chunks per row in one part of K
  rcp::GemvPhase phase[rcp::kMaxPhases];
  int off_bar, off_T0c, off_scale, off_red, off_bs, off_qbuf, off_part;
  int bs_bytes, red_bytes, part_bytes;
  int stage_stride;   // ring stage: boxes of weights, plus the stage's expanded activations when they are streamed
  size_t smem;
};

constexpr size_t kSmemMax = 232448;            // 227 KB of dynamic shared memory per CTA on sm_100
constexpr size_t kExpandBudget = 128 * 1024;   // expanded activations (one byte per code and token) per CTA
constexpr size_t kExpandBudgetTwoTiles = 80 * 1024;   // the same with 9 to 16 tokens (their reduction buffers are larger)

// Tokens one launch can take: their expanded activations must fit beside a ring of three stages.
// cap 16: the tensor-core kernel with two column tiles takes 9 to 16 tokens at once where they fit.
int tokens_per_pass(int M, int K, int cap) {
  if (cap > 8) {
    if (M > 8 && (size_t)M * K <= kExpandBudgetTwoTiles) return M;
    cap = 8;
  }
  int m = std::min(M, cap);
  while (m > 1 && (size_t)m * K > kExpandBudget) m--;
  return m;
}

// The tensor-core kernels of the per-row grid rather keep their (up to eight) tokens and go through K in
// parts when the expanded activations of the whole K would not fit: the weights are then streamed once, not
// once per launch. Falls back to fewer tokens when the sums parked between the parts leave no room for a
// ring of three stages (very many rows per CTA). Returns the tokens per launch, *nsplit the parts of K.
StreamPlan make_plan(int M, int N, int K, int sms, bool grouped = false, size_t qbuf = 0, int nsplit = 1,
                     bool stream_act = false);
int tokens_and_parts(int M, int N, int K, int cap, int sms, int* nsplit) {
  *nsplit = 1;
  const int m = tokens_per_pass(M, K, cap);
  if (cap < 8 || m > 8) return m;
  const int want = std::min(M, 8);
  if (m == want) return m;   // everything fits at once (measured: parts cost more than a ring of two stages does)
  for (int parts = (int)(((size_t)want * K + kExpandBudget - 1) / kExpandBudget); parts <= 8; parts++) {
    const StreamPlan pl = make_plan(want, N, K, sms, false, 0, parts);
    if (pl.stages >= 3 && pl.smem <= kSmemMax) {
      *nsplit = pl.nsplit;
      return want;
    }
  }
  return m;
}

// Cost model of a phase in clocks: stages x (warps sharing a scheduler) x clocks per warp and
// chunk on one of the four schedulers, plus a fixed cost per phase (LUT fetch, reduction, barrier).
long long phase_cost(int gpc, int nchunk) {
  const int KS = rcp::kCWarps / gpc;
  const int stages = (nchunk + KS - 1) / KS;
  const int per_sched = (gpc * KS + 3) / 4;
  return (long long)stages * per_sched * 504 + 2000;
}

// A phase with the quotients the kernel would otherwise divide for.
rcp::GemvPhase make_phase(int gpc, int first, int total, int ncta, int reps, int nchunk, int ks_cap = rcp::kCWarps) {
  rcp::GemvPhase ph;
  ph.gpc = gpc; ph.first = first; ph.total = total; ph.ncta = ncta; ph.reps = reps;
  ph.q = total / ncta;
  ph.r = total % ncta;
  ph.ks = std::min(rcp::kCWarps / gpc, ks_cap);
  ph.inv_ks = (256 + ph.ks - 1) / ph.ks;
  ph.sa = (nchunk + ph.ks - 1) / ph.ks;
  return ph;
}

// Splits `rem` leftover groups (fewer than 16 per CTA) into phases: shares of 8, 4, 2 or 1 groups
// per CTA keep all warps busy but cost a phase each; one last phase takes whatever is left,
// ceil(left / CTAs) groups per CTA. Picks the cheapest combination. Returns the number of phases.
// ks_cap: most warps that may share a group along K (streamed activations: a stage holds the activations of
// that many chunks); phases that would need more are left out, the last phase uses fewer warps per group.
int plan_leftover(int rem, int sms, int nchunk, rcp::GemvPhase* out, int ks_cap = rcp::kCWarps) {
  int best_mask = 0;
  long long best = -1;
  for (int mask = 0; mask < 16; mask++) {   // bit i: a phase of 8 >> i groups per CTA
    int left = rem;
    long long cost = 0;
    bool ok = true;
    for (int i = 0; i < 4; i++) {
      if (!(mask >> i & 1)) continue;
      const int gpc = 8 >> i;
      if (rcp::kCWarps / gpc > ks_cap) { ok = false; break; }
      if (left < gpc * sms) { ok = false; break; }
      left -= gpc * sms;
      cost += phase_cost(gpc, nchunk);
    }
    if (!ok) continue;
    if (left >= 16 * sms) continue;
    if (left > 0) cost += phase_cost((left + sms - 1) / sms, nchunk);
    if (best < 0 || cost < best) { best = cost; best_mask = mask; }
  }
  int n = 0, first = 0, left = rem;
  for (int i = 0; i < 4; i++) {
    if (!(best_mask >> i & 1)) continue;
    const int gpc = 8 >> i;
    out[n++] = make_phase(gpc, first, gpc * sms, sms, 1, nchunk, ks_cap);
    first += gpc * sms;
    left -= gpc * sms;
  }
  if (left > 0) {
    const int ncta = std::min(left, sms);
    out[n++] = make_phase((left + ncta - 1) / ncta, first, left, ncta, 1, nchunk, ks_cap);
  }
  return n;
}

// qbuf: bytes of staging for the fused quantizer's cross-warp rotation strides (0 if unused)
// nsplit: parts of K the kernel goes through one after the other (tensor-core kernels of the per-row grid)
// stream_act: the expanded activations travel with the ring stages (tensor-core kernels of the per-row grid)
// instead of being expanded for the whole K up front.
StreamPlan make_plan(int M, int N, int K, int sms, bool grouped, size_t qbuf, int nsplit, bool stream_act) {
  StreamPlan pl;
  pl.grid = sms;
  pl.nchunk_total = (K / 16 + rcp::kChunkWords - 1) / rcp::kChunkWords;
  pl.nsplit = std::max(1, std::min(nsplit, pl.nchunk_total));
  pl.nchunk = (pl.nchunk_total + pl.nsplit - 1) / pl.nsplit;
  pl.nsplit = (pl.nchunk_total + pl.nchunk - 1) / pl.nchunk;   // no empty part
  // Phases: first the groups left over when every CTA takes 16 per round, then the rounds.
  const int groups = (N + 15) / 16;
  const int per_round = sms * rcp::kCWarps;
  const int R = groups / per_round;
  const int ks_cap = stream_act ? std::max(1, 32 / M) : rcp::kCWarps;
  pl.nphase = plan_leftover(groups - R * per_round, sms, pl.nchunk, pl.phase, ks_cap);
  int first = groups - R * per_round;
  if (R > 0) pl.phase[pl.nphase++] = make_phase(rcp::kCWarps, first, per_round, sms, R, pl.nchunk);
  int ks_max = 1;
  for (int i = 0; i < pl.nphase; i++) ks_max = std::max(ks_max, pl.phase[i].ks);
  // streamed: per stage, 512 bytes per token and chunk of the stage, rounded so that the stages stay 1024-byte aligned
  const size_t bstage = stream_act ? ((size_t)ks_max * M * 512 + 1023) / 1024 * 1024 : 0;
  pl.stage_stride = (int)(rcp::kStageBytes + bstage);
  const size_t bs_bytes = stream_act ? 0 : (size_t)pl.nchunk * rcp::kChunkWords * 16 * M;
  // sums of q per chunk (per group of 128: four per chunk); reduction buffers: integer sums of 8
  // row groups x 3 planes, or (group-wise grid) fp32 terms of every warp, tokens in pairs x 16 rows
  const size_t t0c_bytes = grouped ? (size_t)(M + 1) * pl.nchunk * 16 : (((size_t)M * pl.nchunk * 4) + 15) / 16 * 16;
  const size_t red_bytes = grouped ? (size_t)rcp::kCWarps * ((M + 1) / 2) * 32 * 4 : (size_t)2 * 8 * 16 * M * 3 * 4;
  // K in parts: the integer sums of every group this CTA owns wait in shared memory between the parts
  int own_groups = 0;
  for (int i = 0; i < pl.nphase; i++) own_groups += pl.phase[i].reps * (pl.phase[i].q + (pl.phase[i].r ? 1 : 0));
  const size_t part_bytes = pl.nsplit > 1 ? (size_t)own_groups * 16 * M * 3 * 4 : 0;
  const size_t misc = 128 + t0c_bytes + 256 + red_bytes + qbuf + part_bytes;
  const size_t fixed = 1024 + misc + bs_bytes;
  pl.stages = fixed >= kSmemMax ? 0 : (int)std::min<size_t>(rcp::kMaxStages, (kSmemMax - fixed) / pl.stage_stride);
  size_t off = (size_t)pl.stages * pl.stage_stride;
  pl.off_bar = (int)off; off += 128;
  pl.off_T0c = (int)off; off += t0c_bytes;
  pl.off_scale = (int)off; off += 256;   // 16 scales, 16 per-warp maxima of the fused quantizer, 16 token totals
  pl.off_red = (int)off; off += red_bytes;
  pl.off_bs = (int)off; off += bs_bytes;
  pl.off_qbuf = (int)off; off += qbuf;
  pl.off_part = (int)off; off += part_bytes;
  pl.bs_bytes = (int)bs_bytes; pl.red_bytes = (int)red_bytes; pl.part_bytes = (int)part_bytes;
  pl.smem = off + 1024;
  return pl;
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

constexpr int kMaxDevices = 64;

// Tensor maps of boxes of 16 gpcs[i] rows x 128 bytes (those with a count of 0 repeat the first). Encoding one costs the
// host about a microsecond, so the maps of the last few (weights, shape, boxes) combinations are remembered per thread.
int phase_maps(const uint32_t* words, int N, int K, int nphase, const int* gpcs, const rcp::GemvMaps** out) {   // gpcs [kMaxPhases]
  struct MapKey { const void* words; int N, K, nphase, gpc[rcp::kMaxPhases]; };
  struct MapSlot { MapKey key; rcp::GemvMaps maps; bool used; };
  constexpr int kMapSlots = 16;
  thread_local MapSlot map_cache[kMapSlots] = {};
  thread_local int map_next = 0;
  MapKey key = {};
  key.words = words; key.N = N; key.K = K; key.nphase = nphase;
  for (int i = 0; i < rcp::kMaxPhases; i++) key.gpc[i] = gpcs[i];
  for (int i = 0; i < kMapSlots; i++)
    if (map_cache[i].used && std::memcmp(&map_cache[i].key, &key, sizeof(MapKey)) == 0) { *out = &map_cache[i].maps; return RCP_OK; }
  EncodeTiledFn enc = encode_tiled_fn();
  if (!enc) return cuda_fail(cudaErrorNotSupported);
  MapSlot& slot = map_cache[map_next];
  map_next = (map_next + 1) % kMapSlots;
  slot.used = false;
  const cuuint64_t gdim[2] = {(cuuint64_t)(K / 16), (cuuint64_t)N};
  const cuuint64_t gstride[1] = {(cuuint64_t)(K / 4)};
  const cuuint32_t estr[2] = {1, 1};
  for (int i = 0; i < rcp::kMaxPhases; i++) {
    if (gpcs[i] < 1 && i > 0) { slot.maps.m[i] = slot.maps.m[0]; continue; }
    const int gpc = std::max(1, gpcs[i]);
    const cuuint32_t box[2] = {(cuuint32_t)rcp::kChunkWords, (cuuint32_t)(16 * gpc)};
    const CUresult r = enc(&slot.maps.m[i], CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, const_cast<uint32_t*>(words), gdim,
                           gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return cuda_fail(cudaErrorInvalidValue);
  }
  slot.key = key;
  slot.used = true;
  *out = &slot.maps;
  return RCP_OK;
}

// ---------------------------------------------------------------------------------------------
// GEMV on tcgen05: launch plan.
struct UmmaPlan {
  int tokens;        // that it is made for
  int nchunk, nphase, grid, kpl, lg_kpl, bgroup, bstep, bhalf, lg_m2, slots, dcols, acc_cols, nbuf, stages, helpers;
  rcp::UmmaPhase phase[rcp::kMaxPhases];
  int part_chunks;   // nchunk (rounded up to kpl): all of K at once
  long long clocks;  // estimate of its items
  int off_bar, off_misc, off_red, off_bs, off_qbuf, red_bytes, bs_bytes;
  size_t smem;
};

// Columns of the kind::i8 instructions for kp chunks side by side: a column per token and one of ones for each.
int umma_columns(int M, int kp) {
  const int n = kp * (M + 1);
  return n <= 8 ? 8 : (n + 15) / 16 * 16;
}
// kind::f8f6f4 with 128 rows is specified for multiples of 16 columns alone. (Sixteen for all three: 57344x8192 at three tokens
// 25.6 -> 26.2 us a call, half as many sets of accumulators fitting; for that one alone, no difference.)
int umma_columns_f8(int ncol) { return std::max(16, ncol); }
int floor_pow2(int v) { int p = 1; while (2 * p <= v) p *= 2; return p; }

// stages 0: does not fit. qbuf: bytes of scratch for the quantizer inside.
//   An item takes the longest of: 16 KB of weights for every SM from HBM, 720 clocks (a part of that where fewer lanes are in
// use); its 48 instructions, 600 clocks up to 16 columns, 24 a column from there on; a slot's turn, 860 clocks where the
// accumulators (three times 48 columns) leave room for two slots only. Columns buy lanes (kp chunks side by side), which is
// what short or few rows need; up to 32 or up to 48 of them, whichever comes out cheaper.
UmmaPlan umma_plan_for(int M, int N, int K, int sms, size_t qbuf, int kp_max, int max_cols, bool parts, long long* total) {
  UmmaPlan pl = {};
  pl.tokens = M;
  pl.grid = sms;
  pl.nchunk = (K / 16 + rcp::kChunkWords - 1) / rcp::kChunkWords;
  int kp_cap = kp_max;
  while (kp_cap > 1 && (umma_columns(M, kp_cap) > max_cols || kp_cap >= 2 * pl.nchunk)) kp_cap /= 2;
  auto kp_of = [&](int g) { return std::min(kp_cap, floor_pow2(8 / g)); };
  auto items_of = [&](int g) { return (pl.nchunk + kp_of(g) - 1) / kp_of(g); };
  auto item_of = [&](int g, int hbm) {
    return (long long)std::max(std::max(hbm * g * kp_of(g) / 8, max_cols > 32 ? 860 : 600), 24 * umma_columns(M, kp_of(g)));
  };
  auto cost_of = [&](int g) { return items_of(g) * item_of(g, 720) + 400; };
  const int groups = (N + 15) / 16, per_round = 8 * sms, rounds = groups / per_round, left0 = groups - rounds * per_round;
  *total = 0;
  if (parts && groups > per_round) return pl;   // K in parts: one tile per CTA
  // the groups left over from the rounds of eight per CTA: phases of 4, 2, 1 groups per CTA, and one last for what remains
  int best_mask = 0;
  long long best = -1;
  for (int mask = 0; mask < (parts ? 1 : 8); mask++) {
    int left = left0;
    long long cost = 0;
    bool ok = true;
    for (int i = 0; i < 3; i++) {
      if (!(mask >> i & 1)) continue;
      const int g = 4 >> i;
      if (left < g * sms) { ok = false; break; }
      left -= g * sms;
      cost += cost_of(g);
    }
    if (!ok) continue;
    if (left > 0) cost += cost_of((left + sms - 1) / sms);
    if (best < 0 || cost < best) { best = cost; best_mask = mask; }
  }
  *total = pl.clocks = best + (rounds > 0 ? rounds * cost_of(8) : 0);
  int first = 0;
  auto add = [&](int g, int n, int ncta, int reps) {
    rcp::UmmaPhase& ph = pl.phase[pl.nphase++];
    ph.gpc = g; ph.first = first; ph.total = n; ph.ncta = ncta; ph.reps = reps;
    ph.q = n / ncta; ph.r = n % ncta;
    ph.kp = kp_of(g); ph.items = items_of(g); ph.ncol = umma_columns(M, ph.kp);
    ph.ncol_f8 = umma_columns_f8(ph.ncol);
    ph.inv_rows = (65536 + 16 * g - 1) / (16 * g);
    first += n * reps;
  };
  int left = left0;
  for (int i = 0; i < 3; i++) {
    if (!(best_mask >> i & 1)) continue;
    const int g = 4 >> i;
    add(g, g * sms, sms, 1);
    left -= g * sms;
  }
  if (left > 0) {
    const int ncta = std::min(left, sms);
    add((left + ncta - 1) / ncta, left, ncta, 1);
  }
  if (rounds > 0) add(8, per_round, sms, rounds);
  pl.kpl = 1;
  int ncol = 8;
  for (int i = 0; i < pl.nphase; i++) { pl.kpl = std::max(pl.kpl, pl.phase[i].kp); ncol = std::max(ncol, pl.phase[i].ncol); }
  while ((1 << pl.lg_kpl) < pl.kpl) pl.lg_kpl++;
  while ((1 << pl.lg_m2) < M) pl.lg_m2++;
  pl.dcols = ncol;
  pl.acc_cols = 2 * ncol + umma_columns_f8(ncol);
  pl.slots = pl.acc_cols <= 128 ? 3 : 2;
  pl.nbuf = std::min(rcp::kUMaxBuf, (512 - 128 * pl.slots) / pl.acc_cols);
  // activations: odd strides (in 16 bytes) between the halves and two pieces more between the steps keep the quantizer's
  // narrow stores out of one another's banks
  pl.bhalf = (pl.kpl * (M + 1)) | 1;
  pl.bstep = 8 * pl.bhalf + 2;
  pl.bgroup = 4 * pl.bstep;
  bool shared = false;
  for (int i = 0; i < pl.nphase; i++) shared |= pl.phase[i].kp > 1;
  pl.red_bytes = shared ? M * 3 * rcp::kULanes * 4 : 0;
  const size_t bar_bytes = 8 * (2 * rcp::kUMaxStages + 2 * rcp::kUMaxSlots + 2 * rcp::kUMaxBuf + 3), misc_bytes = 256;
  const size_t fixed = 1024 + bar_bytes + misc_bytes + pl.red_bytes + qbuf + 64 + 16 * umma_columns_f8(ncol);
  // as few parts of K as leave room for three stages (one part: for two)
  for (int n = parts ? 2 : 1; n <= (parts ? 8 : 1); n++) {
    pl.part_chunks = ((pl.nchunk + n - 1) / n + pl.kpl - 1) / pl.kpl * pl.kpl;
    const long long bytes = (long long)(pl.part_chunks / pl.kpl) * pl.bgroup * 16;
    const long long room = (long long)kSmemMax - (long long)fixed - bytes;
    pl.stages = room < 0 ? 0 : (int)std::min<long long>(rcp::kUMaxStages, room / rcp::kUItemBytes);
    pl.bs_bytes = (int)std::min<long long>(bytes + 16 * umma_columns_f8(ncol), 1 << 20);
    if (pl.stages >= (parts ? 3 : 2)) break;
    pl.stages = 0;
  }
  if (!pl.stages) return pl;
  // Two stages do not keep enough requests in flight for 720 clocks an item (12288x20800, us a call: 22.0 at six tokens with three
  // stages, 30.3 at eight with two).
  if (pl.stages == 2)
    for (int i = 0; i < pl.nphase; i++)
      pl.clocks += pl.phase[i].reps * pl.phase[i].items * (item_of(pl.phase[i].gpc, 1100) - item_of(pl.phase[i].gpc, 720));
  // Up to eight tokens are finished by half of the workers; the others help to convert. Two teams want a ring of five stages:
  // a team that waits for a stage's next fill must know that the one before has come, and it does know that of the items five
  // back (their slots were free before it wrote its last).
  pl.helpers = M <= 2 * rcp::kUTok && pl.stages >= 5 && !parts;   // (K in parts: the workers are busy with the next part)
  size_t off = (size_t)pl.stages * rcp::kUItemBytes;
  pl.off_bar = (int)off; off += (bar_bytes + 15) / 16 * 16;
  pl.off_misc = (int)off; off += misc_bytes;
  pl.off_red = (int)off; off += pl.red_bytes;
  pl.off_bs = (int)off; off += pl.bs_bytes;
  pl.off_qbuf = (int)off; off += qbuf;
  pl.smem = off + 1024;
  return pl;
}
// kp_max: most chunks side by side
UmmaPlan make_umma_plan(int M, int N, int K, int sms, size_t qbuf, int kp_max = 8) {
  long long cost[2];
  UmmaPlan a = umma_plan_for(M, N, K, sms, qbuf, kp_max, 32, false, &cost[0]), b = umma_plan_for(M, N, K, sms, qbuf, kp_max, 48, false, &cost[1]);
  if (a.stages && b.stages) return cost[1] < cost[0] ? b : a;
  if (a.stages || b.stages || qbuf || M == 1) return a.stages ? a : b;
  // the activations do not fit: K in parts
  a = umma_plan_for(M, N, K, sms, qbuf, kp_max, 32, true, &cost[0]);
  b = umma_plan_for(M, N, K, sms, qbuf, kp_max, 48, true, &cost[1]);
  return !b.stages || (a.stages && cost[0] <= cost[1]) ? a : b;
}

// SMs of the current device (remembered per device; 148 if the query fails)
int sm_count() {
  static std::mutex mu;
  static int n[kMaxDevices] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 148;
  std::lock_guard<std::mutex> lock(mu);
  if (!n[dev] && cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n[dev] = 148;
  return n[dev];
}

// cudaFuncAttributeMaxDynamicSharedMemorySize belongs to the (kernel, device) pair: set once per device (mu and done
// belong to the kernel)
template <typename Kern>
cudaError_t set_max_smem(Kern kern, int bytes, std::mutex& mu, bool (&done)[kMaxDevices]) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!done[dev]) {
    const cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (r != cudaSuccess) return r;
    done[dev] = true;
  }
  return cudaSuccess;
}

template <int MODE, int MTOK, bool GRP, int FQ, bool A16, bool SPLIT, bool SDBG, bool SB, bool LATE>
int launch_stream_k(const rcp::GemvMaps& maps, const rcp::GemvParams& gp, const StreamPlan& pl, cudaStream_t st) {
  // cudaFuncAttributeMaxDynamicSharedMemorySize belongs to the (kernel, device) pair: set once per device
  static std::mutex mu;
  static bool attr_set[kMaxDevices] = {};
  auto kern = rcp::gemv_stream_kernel<MODE, MTOK, GRP, FQ, A16, SPLIT, SDBG, SB, LATE>;
  int dev = 0;
  RCP_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return RCP_ERR_LIMIT;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (!attr_set[dev]) {
      RCP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
      attr_set[dev] = true;
    }
  }
  RCP_CUDA(launch_overlapped(kern, dim3(pl.grid), dim3(SB ? rcp::kGThreads + 32 * rcp::kExpWarps : rcp::kGThreads), pl.smem, st, maps, gp));
  return RCP_OK;
}

// late: which of its two forms a tensor-core kernel is taken in. (The checked instantiations have the
// early form alone; digit columns of more than one token always have the kernel that splits them in front: late.)
template <int MODE, int MTOK, bool GRP, int FQ, bool A16, bool SPLIT, bool SDBG, bool SB = false>
int launch_stream_s(const rcp::GemvMaps& maps, const rcp::GemvParams& gp, const StreamPlan& pl, bool late, cudaStream_t st) {
  constexpr bool kBoth = MODE == rcp::kModeMma && !SDBG, kAlways = kBoth && A16 && (SPLIT || MTOK == 16);
  if constexpr (kAlways) {
    return launch_stream_k<MODE, MTOK, GRP, FQ, A16, SPLIT, SDBG, SB, true>(maps, gp, pl, st);
  } else {
    if constexpr (kBoth)
      if (late) return launch_stream_k<MODE, MTOK, GRP, FQ, A16, SPLIT, SDBG, SB, true>(maps, gp, pl, st);
    return launch_stream_k<MODE, MTOK, GRP, FQ, A16, SPLIT, SDBG, SB, false>(maps, gp, pl, st);
  }
}

// streamed activations (tensor-core kernels of the per-row grid; MTOK 0: up to eight tokens, 16: nine to sixteen)
template <int MTOK>
int launch_stream_sb(const rcp::GemvMaps& maps, const rcp::GemvParams& gp, const StreamPlan& pl, bool late, cudaStream_t st) {
  if (gp.S_out) return launch_stream_s<rcp::kModeMma, MTOK, false, 0, false, false, true, true>(maps, gp, pl, late, st);
  return launch_stream_s<rcp::kModeMma, MTOK, false, 0, false, false, false, true>(maps, gp, pl, late, st);
}

// gp.S_out set: the checked instantiation of the same kernel, which also stores its integer sums.
template <int MODE, int MTOK, bool GRP = false, int FQ = 0, bool A16 = false, bool SPLIT = false>
int launch_stream_t(const rcp::GemvMaps& maps, const rcp::GemvParams& gp, const StreamPlan& pl, bool late, cudaStream_t st) {
  if (gp.S_out) return launch_stream_s<MODE, MTOK, GRP, FQ, A16, SPLIT, true>(maps, gp, pl, late, st);
  return launch_stream_s<MODE, MTOK, GRP, FQ, A16, SPLIT, false>(maps, gp, pl, late, st);
}

// One launch: M tokens (their expanded activations fit in shared memory). grouped: lut_f16 is
// [N][K/128][4], one grid per group of 128 weights.
// Activations still to be rotated and quantized, for the kernels that do it themselves.
struct FusedAct {
  const void* x_f16;     // [M][K]
  int B;                 // rotation block, 1 = none
  float clip_ratio;
  uint8_t* xq_out;       // optional
  void* scale_out;       // optional
};

// Weight-only form, activations still in fp16: the GEMV kernel makes the digit planes itself.
struct SplitAct {
  const void* x_f16;    // [tokens][K]
  int8_t* digits_out;   // [tokens][4][K], written by CTA 0
  float* unit_out;      // [tokens][4], written by CTA 0
};

// Shapes the in-kernel quantizer takes: one token under one rotation block of 2048, 4096 or 8192 elements, or in blocks
// of at most 512 with K up to 16384. Measured on B200, us a call in a chain of calls, cold weights, two kernels -> one:
// 2048x2048 3.8 -> 2.9, 4096x4096 5.0 -> 4.05, 57344x8192 32.6 -> 30.7, 333x5184 4.5 -> 3.5, 4096x14336 8.95 -> 8.0.
// At K = 28672 (four words per thread) the stand-alone quantizer's cluster of eight CTAs is faster than all CTAs doing
// the whole token (8192x28672 21.6 -> 22.3), and two tokens are twice the serial work.
bool full_block(int K, int B) { return B == K && (K == 2048 || K == 4096 || K == 8192); }
bool fused_ok(int M, int K, int B) { return M == 1 && (full_block(K, B) || (B <= 512 && K <= 16384)); }

template <bool GRP>
int launch_fused(const rcp::GemvMaps& maps, const rcp::GemvParams& gp, const StreamPlan& pl, bool late, cudaStream_t st) {
  if (full_block(gp.K, gp.had_block)) {
    if (gp.K == 2048) return launch_stream_t<rcp::kModeDp4a, 1, GRP, 4>(maps, gp, pl, late, st);
    if (gp.K == 4096) return launch_stream_t<rcp::kModeDp4a, 1, GRP, 8>(maps, gp, pl, late, st);
    return launch_stream_t<rcp::kModeDp4a, 1, GRP, 16>(maps, gp, pl, late, st);
  }
  if (gp.K <= 8192) return launch_stream_t<rcp::kModeDp4a, 1, GRP, -1>(maps, gp, pl, late, st);
  return launch_stream_t<rcp::kModeDp4a, 1, GRP, -2>(maps, gp, pl, late, st);
}

int launch_stream(int mode, const uint32_t* words, const void* lut_f16, const uint8_t* xq, const void* scale_f16,
                  int M, int N, int K, void* y_f16, void* workspace, cudaStream_t st, bool grouped = false,
                  const FusedAct* fa = nullptr, const float* unit = nullptr, int nsplit = 1,
                  const SplitAct* sa = nullptr, int32_t* S_out = nullptr, bool stream_act = false, bool late = false) {
  if (stream_act && (mode != rcp::kModeMma || fa || unit || sa || nsplit > 1 || M > (grouped ? 8 : rcp::kMaxTokens))) return RCP_ERR_VARIANT;
  if (nsplit > 1 && (mode != rcp::kModeMma || grouped || fa || M > 8)) return RCP_ERR_VARIANT;
  if (sa && (mode != rcp::kModeMma || grouped || fa || unit || nsplit > 1 || M != 4 || K > 16384)) return RCP_ERR_VARIANT;
  // unit: weight-only form; xq then holds M digit columns of K signed bytes (four per token), scale_f16 is unused
  if (unit && (mode != rcp::kModeMma || grouped || fa || M % 4)) return RCP_ERR_VARIANT;
  if (mode != rcp::kModeMma && M > 2) return RCP_ERR_VARIANT;
  if (M > 8 && (grouped || fa || M > rcp::kMaxTokens)) return RCP_ERR_VARIANT;
  if (grouped && (mode == rcp::kModeHybrid || K % 128)) return RCP_ERR_VARIANT;
  if (fa && (mode != rcp::kModeDp4a || !fused_ok(M, K, fa->B))) return RCP_ERR_VARIANT;
  // The plan depends on sizes and form alone; working it out costs the host a quarter of a microsecond, so the last few
  // are remembered per thread.
  struct PlanKey { size_t qbuf; int M, N, K, sms, nsplit, grouped, stream_act, unused; };   // (no padding: compared as bytes)
  struct PlanSlot { PlanKey key; StreamPlan plan; };
  constexpr int kPlanSlots = 16;
  thread_local PlanSlot plan_cache[kPlanSlots] = {};   // (M is 0 in an unused slot)
  thread_local int plan_next = 0;
  PlanKey pk = {};
  pk.M = M; pk.N = N; pk.K = K; pk.sms = sm_count(); pk.nsplit = nsplit; pk.grouped = grouped; pk.stream_act = stream_act;
  pk.qbuf = fa ? (full_block(K, fa->B) ? rcp::full_rotate_bytes(K) : 0) : (sa ? (size_t)M * K : 0);
  const StreamPlan* found = nullptr;
  for (int i = 0; i < kPlanSlots && !found; i++)
    if (std::memcmp(&plan_cache[i].key, &pk, sizeof(PlanKey)) == 0) found = &plan_cache[i].plan;
  if (!found) {
    PlanSlot& slot = plan_cache[plan_next];
    plan_next = (plan_next + 1) % kPlanSlots;
    slot.plan = make_plan(M, N, K, pk.sms, grouped, pk.qbuf, nsplit, stream_act);
    slot.key = pk;
    found = &slot.plan;
  }
  const StreamPlan& pl = *found;
  if (pl.stages < 2 || pl.smem > kSmemMax) return RCP_ERR_SHAPE;
  int gpc[rcp::kMaxPhases] = {};
  for (int i = 0; i < pl.nphase; i++) gpc[i] = pl.phase[i].gpc;
  const rcp::GemvMaps* cached = nullptr;
  const int rc_maps = phase_maps(words, N, K, pl.nphase, gpc, &cached);
  if (rc_maps != RCP_OK) return rc_maps;
  const rcp::GemvMaps& maps = *cached;
  rcp::GemvParams gp;
  gp.lut = static_cast<const uint2*>(lut_f16);
  gp.xq = xq;
  gp.scale = static_cast<const __half*>(scale_f16);
  gp.unit = unit;
  gp.y = static_cast<__half*>(y_f16);
  gp.status = static_cast<int32_t*>(workspace);
  gp.S_out = S_out;
  gp.M = M; gp.N = N; gp.K = K;
  gp.ngrp = grouped ? K / 128 : 0;
  gp.nchunk = pl.nchunk;
  gp.nchunk_total = pl.nchunk_total;
  gp.nsplit = pl.nsplit;
  gp.off_part = pl.off_part;
  gp.act_parts = std::max(1, rcp::kCWarps / M);
  gp.inv_act_parts = (256 + gp.act_parts - 1) / gp.act_parts;
  gp.nphase = pl.nphase;
  for (int i = 0; i < rcp::kMaxPhases; i++) gp.phase[i] = i < pl.nphase ? pl.phase[i] : make_phase(1, 0, 0, 1, 0, pl.nchunk);
  gp.stages = pl.stages;
  // one 32 KB stage per CTA at about 6 TB/s for the whole grid, in SM clocks (about 2 GHz)
  gp.ramp_clk = (int)((double)rcp::kStageBytes * pl.grid / 6.0e12 * 1.9e9);
  gp.off_bar = pl.off_bar; gp.off_T0c = pl.off_T0c; gp.off_scale = pl.off_scale; gp.off_red = pl.off_red;
  gp.off_bs = pl.off_bs;
  gp.bs_bytes = pl.bs_bytes; gp.red_bytes = pl.red_bytes; gp.part_bytes = pl.part_bytes;
  gp.stage_stride = pl.stage_stride;
  gp.off_qbuf = pl.off_qbuf;
  gp.x = nullptr; gp.xq_out = nullptr; gp.scale_out = nullptr; gp.unit_out = nullptr;
  gp.inv_sqrt_b = 1.f; gp.clip_ratio = 1.f; gp.had_block = 1;
  if (fa) {
    gp.x = static_cast<const __half*>(fa->x_f16);
    gp.xq_out = fa->xq_out;
    gp.scale_out = static_cast<__half*>(fa->scale_out);
    gp.inv_sqrt_b = (float)(1.0 / std::sqrt((double)fa->B));
    gp.clip_ratio = std::min(fa->clip_ratio, rcp::kClipRatioCap);
    gp.had_block = fa->B;
    return grouped ? launch_fused<true>(maps, gp, pl, late, st) : launch_fused<false>(maps, gp, pl, late, st);
  }
  if (sa) {
    gp.x = static_cast<const __half*>(sa->x_f16);
    gp.xq_out = reinterpret_cast<uint8_t*>(sa->digits_out);
    gp.unit_out = sa->unit_out;
    return launch_stream_t<rcp::kModeMma, 0, false, 0, true>(maps, gp, pl, late, st);
  }
  if (unit) {
    if (pl.nsplit > 1) return launch_stream_t<rcp::kModeMma, 0, false, 0, true, true>(maps, gp, pl, late, st);
    return M > 8 ? launch_stream_t<rcp::kModeMma, 16, false, 0, true>(maps, gp, pl, late, st)
                 : launch_stream_t<rcp::kModeMma, 0, false, 0, true>(maps, gp, pl, late, st);
  }
  if (grouped) {
    if (mode == rcp::kModeDp4a)
      return M == 1 ? launch_stream_t<rcp::kModeDp4a, 1, true>(maps, gp, pl, late, st)
                    : launch_stream_t<rcp::kModeDp4a, 2, true>(maps, gp, pl, late, st);
    if (stream_act)
      return gp.S_out ? launch_stream_s<rcp::kModeMma, 0, true, 0, false, false, true, true>(maps, gp, pl, late, st)
                      : launch_stream_s<rcp::kModeMma, 0, true, 0, false, false, false, true>(maps, gp, pl, late, st);
    if (M == 8 && !gp.S_out) return launch_stream_s<rcp::kModeMma, 8, true, 0, false, false, false>(maps, gp, pl, late, st);
    return launch_stream_t<rcp::kModeMma, 0, true>(maps, gp, pl, late, st);
  }
  if (mode == rcp::kModeHybrid)
    return M == 1 ? launch_stream_t<rcp::kModeHybrid, 1>(maps, gp, pl, late, st)
                  : launch_stream_t<rcp::kModeHybrid, 2>(maps, gp, pl, late, st);
  if (mode == rcp::kModeDp4a)
    return M == 1 ? launch_stream_t<rcp::kModeDp4a, 1>(maps, gp, pl, late, st)
                  : launch_stream_t<rcp::kModeDp4a, 2>(maps, gp, pl, late, st);
  if (stream_act) {
    if (M == 8 && !gp.S_out) return launch_stream_sb<8>(maps, gp, pl, late, st);
    return M > 8 ? launch_stream_sb<16>(maps, gp, pl, late, st) : launch_stream_sb<0>(maps, gp, pl, late, st);
  }
  if (pl.nsplit > 1 && M == 8 && !gp.S_out) return launch_stream_s<rcp::kModeMma, 8, false, 0, false, true, false>(maps, gp, pl, late, st);
  if (pl.nsplit > 1) return launch_stream_t<rcp::kModeMma, 0, false, 0, false, true>(maps, gp, pl, late, st);
  if (M == 8 && !gp.S_out) return launch_stream_s<rcp::kModeMma, 8, false, 0, false, false, false>(maps, gp, pl, late, st);   // token count known at compile time
  return M > 8 ? launch_stream_t<rcp::kModeMma, 16>(maps, gp, pl, late, st) : launch_stream_t<rcp::kModeMma, 0>(maps, gp, pl, late, st);
}

template <int FQ, bool SDBG, bool LATE, bool PARTS = false>
int launch_umma_k(const rcp::GemvMaps& maps, const rcp::UmmaParams& up, const UmmaPlan& pl, cudaStream_t st) {
  static std::mutex mu;
  static bool attr_set[kMaxDevices] = {};
  auto kern = rcp::gemv_umma_kernel<FQ, SDBG, LATE, PARTS>;
  RCP_CUDA(set_max_smem(kern, (int)kSmemMax, mu, attr_set));
  RCP_CUDA(launch_overlapped(kern, dim3(pl.grid), dim3(rcp::kUThreads), pl.smem, st, maps, up));
  return RCP_OK;
}
template <int FQ>
int launch_umma_f(const rcp::GemvMaps& maps, const rcp::UmmaParams& up, const UmmaPlan& pl, cudaStream_t st) {
  return up.S_out ? launch_umma_k<FQ, true, false>(maps, up, pl, st) : launch_umma_k<FQ, false, false>(maps, up, pl, st);
}

// What the host works out for a call of M tokens, see umma_choose.
struct UmmaChoice { UmmaPlan plan, last; int tokens, launches; bool faster, faster_late; };   // late: behind a quantizer of its own

// Whether the tcgen05 kernel is the faster one, its host-side plan against the streaming kernel's. In clocks of an SM: the
// streaming kernels take 77 a KB of weights for one token, 80 for up to eight, 171 for sixteen in one launch; the tcgen05
// kernel what its plan adds up to. Against that it starts and ends slower by what a call with little to stream shows (the
// conversion, three instruction streams and the sums' way back through tensor memory lie on its path, and there is more
// code to fetch; one token, whose calls are otherwise launches of one and the same kernel, most: layers of 54144x4096, 4447x896
// and 1920x14336 took 55.9 -> 56.6 with the first of them here). us a linear call in a chain, streaming -> tcgen05: one token
// 4096x4096 3.9 -> 5.2, 10240x8192 9.9 -> 9.5, 57344x8192 30.5 -> 24.8; three 10007x4096 8.3 -> 8.8, 10240x8192 13.3 -> 11.8,
// 57344x8192 39.7 -> 28.1; eight 22016x4096 12.3 -> 13.4, 8192x28672 31.3 -> 28.5, 57344x8192 38.8 -> 31.2; sixteen 6144x4096
// 9.7 -> 11.3, 12288x4096 14.7 -> 12.1, 28672x4096 23.7 -> 16.8, 57344x8192 75.7 -> 40.1.
// Up to eight tokens it also prepares their activations more slowly than the streaming kernels: all of K before the first
// instruction, and behind a quantizer (`late`) nothing hides that, least of all behind the clusters that quantize long tokens
// (a linear call takes up to 5.4 us longer than the plain one there, 2.7 on the streaming kernels; four tokens and more, or tokens a
// power of two apart). Hence a second comparison with a charge that grows with tokens x channels, where going through K in parts
// costs the streaming kernels 4500 clocks each. Set from 800 shapes of 1 to 90000 rows (a linear call, streaming -> tcgen05: 2368x28672 at
// three tokens 11.4 -> 13.1, 5000x24576 at six 22.0 -> 25.4, 5000x40960 at eight 34.5 -> 38.4, 10240x12288 at five 16.5 -> 18.4, which stay on the
// streaming kernels; 9001x28672 at three 25.4 -> 20.9, at eight 31.2 -> 28.8, 12288x14336 at four 20.7 -> 19.0, which do not). Without it the
// worst of them took 1.15 times as long; with it none takes more than 1.03.
bool umma_faster(int M, int N, int K, int sms, const UmmaChoice& c, bool late) {
  int nsplit = 1;
  const int ms = M == 1 ? 1 : tokens_and_parts(M, N, K, 16, sms, &nsplit);
  const long long kb = (long long)(((N + 15) / 16 + sms - 1) / sms) * K / 256;   // of the CTA with the most rows
  const long long per_launch = 2500, streaming = (M + ms - 1) / ms * (kb * (M == 1 ? 77 : ms <= 8 ? 80 : 171) + per_launch);
  const long long slower = M == 1 ? 11000 : M <= 3 ? 3000 : M <= 8 ? 6000 : 7200;
  const long long own = c.launches * (c.plan.clocks + per_launch), mk = (long long)M * K;
  if (own + slower >= streaming) return false;
  if (M == 1 || M > 8) return true;
  if (!late) return own + 3000 + mk * 2 / 100 < streaming;
  const int cluster = K > 8192 && (M > 3 || (K & (K - 1)) == 0) ? 2000 : 0;
  return own + 2000 + mk * 7 / 100 + cluster < streaming + (nsplit <= 4 ? (nsplit - 1) * 4500 : 0);
}

// A call of M tokens: launches of `tokens` of them each (as many as fit beside a ring of two
// stages) by `plan`, the last one with what remains by `last` (0 launches: not even one token fits), and whether that is
// faster than the streaming kernels.
void umma_choose(int M, int N, int K, int sms, size_t qbuf, UmmaChoice& c) {
  c.tokens = c.launches = 0;
  c.faster = c.faster_late = false;
  for (int parts = 1; parts <= M && !c.launches; parts++) {
    const int m = (M + parts - 1) / parts, n = (M + m - 1) / m, rest = M - (n - 1) * m;
    c.plan = make_umma_plan(m, N, K, sms, qbuf);
    if (!c.plan.stages) continue;
    // What remains may fit only with no more chunks side by side than the others have: fewer tokens would take more, and K is
    // padded to a multiple of them.
    c.last = rest == m ? c.plan : make_umma_plan(rest, N, K, sms, qbuf);
    for (int kp = c.plan.kpl; kp >= 1 && !c.last.stages; kp /= 2) c.last = make_umma_plan(rest, N, K, sms, qbuf, kp);
    if (!c.last.stages) continue;
    c.tokens = m;
    c.launches = n;
  }
  if (c.launches) {
    c.faster = umma_faster(M, N, K, sms, c, false);
    c.faster_late = umma_faster(M, N, K, sms, c, true);
  }
}
// The same, remembered per thread like the streaming kernels' plans.
const UmmaChoice& umma_choice(int M, int N, int K, size_t qbuf) {
  struct Key { size_t qbuf; int M, N, K, sms; };
  struct Slot { Key key; UmmaChoice choice; };
  constexpr int kSlots = 32;
  thread_local Slot cache[kSlots] = {};   // (M is 0 in an unused slot)
  thread_local int next = 0, last = 0;
  Key k = {};
  k.qbuf = qbuf; k.M = M; k.N = N; k.K = K; k.sms = sm_count();
  if (std::memcmp(&cache[last].key, &k, sizeof(Key)) == 0) return cache[last].choice;
  for (int i = 0; i < kSlots; i++)
    if (std::memcmp(&cache[i].key, &k, sizeof(Key)) == 0) { last = i; return cache[i].choice; }
  last = next;
  Slot& slot = cache[next];
  next = (next + 1) % kSlots;
  slot.key = k;
  umma_choose(M, N, K, k.sms, qbuf, slot.choice);
  return slot.choice;
}

// One launch of the tcgen05 kernel by the plan pl. fa: one token still to be rotated and quantized (xq and scale unused).
int launch_umma(const uint32_t* words, const void* lut_f16, const uint8_t* xq, const void* scale_f16, int M, int N, int K,
                void* y_f16, void* workspace, cudaStream_t st, const UmmaPlan& pl, const FusedAct* fa, int32_t* S_out, bool late) {
  if (pl.tokens != M || pl.stages < 2 || pl.smem > kSmemMax) return RCP_ERR_SHAPE;   // (never: the layout is made for so many tokens)
  int gpc[rcp::kMaxPhases] = {};
  for (int i = 0; i < pl.nphase; i++) {   // (five phases at most)
    gpc[i] = pl.phase[i].gpc;
    if (pl.phase[i].r > 0) gpc[rcp::kMaxPhases - 1] = pl.phase[i].gpc - 1;
  }
  const rcp::GemvMaps* maps = nullptr;
  const int rc = phase_maps(words, N, K, pl.nphase, gpc, &maps);
  if (rc != RCP_OK) return rc;
  rcp::UmmaParams up;
  up.lut = static_cast<const uint2*>(lut_f16);
  up.xq = xq;
  up.scale = static_cast<const __half*>(scale_f16);
  up.y = static_cast<__half*>(y_f16);
  up.status = static_cast<int32_t*>(workspace);
  up.S_out = S_out;
  up.M = M; up.N = N; up.K = K; up.nchunk = pl.nchunk; up.nphase = pl.nphase;
  for (int i = 0; i < rcp::kMaxPhases; i++) up.phase[i] = pl.phase[i];
  up.kpl = pl.kpl; up.lg_kpl = pl.lg_kpl; up.bgroup = pl.bgroup; up.bstep = pl.bstep; up.bhalf = pl.bhalf; up.lg_m2 = pl.lg_m2; up.helpers = pl.helpers; up.part_chunks = pl.part_chunks;
  up.slots = pl.slots; up.dcols = pl.dcols; up.acc_cols = pl.acc_cols; up.nbuf = pl.nbuf; up.stages = pl.stages;
  // one item per CTA at about 6 TB/s for the whole grid, in SM clocks (about 2 GHz)
  up.ramp_clk = (int)((double)rcp::kUItemBytes * pl.grid / 6.0e12 * 1.9e9);
  up.off_bar = pl.off_bar; up.off_misc = pl.off_misc; up.off_red = pl.off_red; up.off_bs = pl.off_bs; up.off_qbuf = pl.off_qbuf;
  up.red_bytes = pl.red_bytes; up.bs_bytes = pl.bs_bytes;
  up.x = nullptr; up.xq_out = nullptr; up.scale_out = nullptr;
  up.inv_sqrt_b = 1.f; up.clip_ratio = 1.f; up.had_block = 1;
  if (fa) {
    up.x = static_cast<const __half*>(fa->x_f16);
    up.xq_out = fa->xq_out;
    up.scale_out = static_cast<__half*>(fa->scale_out);
    up.inv_sqrt_b = (float)(1.0 / std::sqrt((double)fa->B));
    up.clip_ratio = std::min(fa->clip_ratio, rcp::kClipRatioCap);
    up.had_block = fa->B;
    if (full_block(K, fa->B)) {
      if (K == 2048) return launch_umma_f<4>(*maps, up, pl, st);
      if (K == 4096) return launch_umma_f<8>(*maps, up, pl, st);
      return launch_umma_f<16>(*maps, up, pl, st);
    }
    return K <= 8192 ? launch_umma_f<-1>(*maps, up, pl, st) : launch_umma_f<-2>(*maps, up, pl, st);
  }
  if (pl.part_chunks < pl.nchunk) {
    if (S_out) return launch_umma_k<0, true, false, true>(*maps, up, pl, st);
    return late ? launch_umma_k<0, false, true, true>(*maps, up, pl, st) : launch_umma_k<0, false, false, true>(*maps, up, pl, st);
  }
  if (S_out) return launch_umma_k<0, true, false>(*maps, up, pl, st);
  return late ? launch_umma_k<0, false, true>(*maps, up, pl, st) : launch_umma_k<0, false, false>(*maps, up, pl, st);
}

int launch_umma_passes(const uint32_t* words, const void* lut_f16, const uint8_t* xq, const void* scale_f16, int M, int N, int K,
                       void* y_f16, void* workspace, cudaStream_t st, int32_t* S_out, bool late) {
  const UmmaChoice& c = umma_choice(M, N, K, 0);
  if (!c.launches) return RCP_ERR_VARIANT;
  for (int i = 0, m0 = 0; i < c.launches; i++, m0 += c.tokens) {
    const int rc = launch_umma(words, lut_f16, xq + (size_t)m0 * (K / 2), static_cast<const __half*>(scale_f16) + m0,
                               std::min(c.tokens, M - m0), N, K, static_cast<__half*>(y_f16) + (size_t)m0 * N, workspace, st,
                               i + 1 < c.launches ? c.plan : c.last, nullptr,
                               S_out ? S_out + (size_t)m0 * N * 4 : nullptr, late);
    if (rc != RCP_OK) return rc;
  }
  return RCP_OK;
}

// All M tokens: as many launches as it takes for the expanded activations to fit (`cap` tokens at most each).
int launch_stream_passes(int mode, int cap, const uint32_t* words, const void* lut_f16, const uint8_t* xq,
                         const void* scale_f16, int M, int N, int K, void* y_f16, void* workspace, cudaStream_t st,
                         bool grouped = false, int32_t* S_out = nullptr, bool late_start = false) {
  int nsplit = 1;
  const int mp = (grouped || cap < 8) ? tokens_per_pass(M, K, cap) : tokens_and_parts(M, N, K, cap, sm_count(), &nsplit);
  // Where the launch would have to go through K in more than four parts (several tokens, a very long K), the form that
  // streams the activations beside the weights is faster: it expands them once per phase, but chunk by chunk among the mask
  // arithmetic, where parts pay a barrier, a fill of the ring's first stage and a set of parked sums each. Measured at eight
  // tokens, parts against streamed: 8192x28672 (three) 28.7 and 31.6 us, 8192x40960 (four) 37.8 and 42.9, 8192x65536 (six)
  // 67.2 and 57.3.
  if (mode == rcp::kModeMma && !grouped && nsplit > 4 && mp == std::min(M, 8)) {
    const StreamPlan sp = make_plan(mp, N, K, sm_count(), false, 0, 1, true);
    if (sp.stages >= 3 && sp.smem <= kSmemMax) {
      for (int m0 = 0; m0 < M; m0 += mp) {
        const int mm = std::min(mp, M - m0);
        const int rc = launch_stream(mode, words, lut_f16, xq + (size_t)m0 * (K / 2),
                                     static_cast<const __half*>(scale_f16) + m0, mm, N, K,
                                     static_cast<__half*>(y_f16) + (size_t)m0 * N, workspace, st, false, nullptr, nullptr, 1,
                                     nullptr, S_out ? S_out + (size_t)m0 * N * 4 : nullptr, true, late_start);
        if (rc != RCP_OK) return rc;
      }
      return RCP_OK;
    }
  }
  // Group-wise grid on the tensor cores, a K so long that not even eight tokens' expanded activations fit: the form
  // with the activations streamed beside the weights takes up to eight tokens in one pass over the weights
  // (8192 x 28672 at eight tokens: one launch instead of two of four tokens).
  if (mode == rcp::kModeMma && grouped && mp < std::min(M, 8)) {
    const int m8 = std::min(M, 8);
    const StreamPlan sp = make_plan(m8, N, K, sm_count(), true, 0, 1, true);
    if (sp.stages >= 3 && sp.smem <= kSmemMax) {
      for (int m0 = 0; m0 < M; m0 += m8) {
        const int mm = std::min(m8, M - m0);
        const int rc = launch_stream(mode, words, lut_f16, xq + (size_t)m0 * (K / 2),
                                     static_cast<const __half*>(scale_f16) + m0, mm, N, K,
                                     static_cast<__half*>(y_f16) + (size_t)m0 * N, workspace, st, true, nullptr, nullptr, 1,
                                     nullptr, S_out ? S_out + (size_t)m0 * N * 4 * (K / 128) : nullptr, true, late_start);
        if (rc != RCP_OK) return rc;
      }
      return RCP_OK;
    }
  }
  for (int m0 = 0; m0 < M; m0 += mp) {
    const int mm = std::min(mp, M - m0);
    int md = mode;
    if (md == rcp::kModeHybrid && mm > 2) md = rcp::kModeMma;
    const int rc = launch_stream(md, words, lut_f16, xq + (size_t)m0 * (K / 2),
                                 static_cast<const __half*>(scale_f16) + m0, mm, N, K,
                                 static_cast<__half*>(y_f16) + (size_t)m0 * N, workspace, st, grouped, nullptr, nullptr,
                                 md == rcp::kModeMma ? nsplit : 1, nullptr,
                                 S_out ? S_out + (size_t)m0 * N * 4 * (grouped ? K / 128 : 1) : nullptr, false, late_start);
    if (rc != RCP_OK) return rc;
  }
  return RCP_OK;
}

// ---------------------------------------------------------------------------------------------
// Scratch of rcp_gemv_w2a4_static: part of the device image, one copy per GPU that loads the library.
static __device__ __align__(256) unsigned char g_static_scratch[RCP_STATIC_SCRATCH_BYTES];

// Device address of g_static_scratch on the current device. In host code the array's name only
// stands for the symbol; the address a kernel can use comes from cudaGetSymbolAddress, asked once
// per device with that device current and remembered afterwards.
int static_scratch_address(void** out) {
  static std::mutex mu;
  static void* addr[kMaxDevices] = {};
  int dev = 0;
  RCP_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return RCP_ERR_LIMIT;
  std::lock_guard<std::mutex> lock(mu);
  if (!addr[dev]) {
    void* p = nullptr;
    RCP_CUDA(cudaGetSymbolAddress(&p, g_static_scratch));
    addr[dev] = p;
  }
  *out = addr[dev];
  return RCP_OK;
}

// Whether one CTA takes a whole token (quantize_act_rows_kernel, quantize_act_full_rows_kernel) or a cluster shares it.
// Measured on B200, cluster -> one CTA, us a call in a chain of them. One block over the token: one CTA at any count
// (K = 4096: 2.7 -> 1.7 for one token, 26 -> 10.8 for 2048). Blocks inside a warp: one CTA up to K = 8192 (8064: 2.7 -> 2.0
// and 34 -> 14.6), above that once the tokens fill the GPU better than eight CTAs each would: 11008 and 14336 even at
// 24 tokens (14336: 2.8 -> 3.6 at 16, 4.2 -> 3.2 at 32, 74 -> 25.8 at 2048), 28672 at 40 (4.7 -> 5.7 at 32, 8.0 -> 5.2
// at 64, 177 -> 50.5 at 2048).
bool rows_form(int M, int K, int B) {
  if (B > 512) return B == K && (K == 2048 || K == 4096 || K == 8192);
  return K <= 8192 || (K <= 16384 && M >= 24) || (K <= 32768 && M >= 40);
}

template <int NT>
int launch_full_rows(const rcp::QuantParams& qp, int M, cudaStream_t st) {
  static std::mutex mu;
  static bool attr_set[kMaxDevices] = {};
  auto kern = rcp::quantize_act_full_rows_kernel<NT>;
  RCP_CUDA(set_max_smem(kern, (int)rcp::full_rows_smem<NT>(), mu, attr_set));
  const int grid = std::min(M, sm_count() * (rcp::kFullRowsThreads / NT));
  RCP_CUDA(launch_overlapped(kern, dim3(grid), dim3(NT), rcp::full_rows_smem<NT>(), st, qp, M));
  return RCP_OK;
}

template <int R, int T_MAX, int BLOCK>
int launch_block_rows(const rcp::QuantParams& qp, int M, cudaStream_t st) {
  static std::mutex mu;
  static bool attr_set[kMaxDevices] = {};
  auto kern = rcp::quantize_act_rows_kernel<R, T_MAX, BLOCK>;
  RCP_CUDA(set_max_smem(kern, R * T_MAX * 32, mu, attr_set));
  const int T = ((qp.K / 16 + R - 1) / R + 31) / 32 * 32;
  const int grid = std::min(M, sm_count() * std::max(1, 1024 / T));
  RCP_CUDA(launch_overlapped(kern, dim3(grid), dim3(T), (size_t)R * T * 32, st, qp, M));
  return RCP_OK;
}

int launch_quantize_rows(const rcp::QuantParams& qp, int M, cudaStream_t st) {
  if (qp.B > 512) {
    if (qp.K == 2048) return launch_full_rows<128>(qp, M, st);
    if (qp.K == 4096) return launch_full_rows<256>(qp, M, st);
    return launch_full_rows<512>(qp, M, st);
  }
  const int W = qp.K / 16;
  if (qp.B == 128) {
    if (W <= 512) return launch_block_rows<1, 512, 128>(qp, M, st);
    // up to one token per SM a thread per word (14336, 96 tokens: 3.6 us against 4.9 with two words per thread), beyond
    // that two smaller CTAs per SM (2048 tokens, with an earlier form of the kernel: 28.5 against 30.0)
    if (W <= 1024 && M <= sm_count()) return launch_block_rows<1, 1024, 128>(qp, M, st);
    if (W <= 896) return launch_block_rows<2, 448, 128>(qp, M, st);
    return launch_block_rows<2, 1024, 128>(qp, M, st);
  }
  return W <= 512 ? launch_block_rows<1, 512, 0>(qp, M, st) : launch_block_rows<2, 1024, 0>(qp, M, st);
}

// Shared memory of which r CTAs fit on an SM (228 KB, 1 KB of it per CTA for the system) and r + 1 do not.
constexpr size_t smem_for_residency(int r) { return 228 * 1024 / (r + 1) - 768; }

// C CTAs per token as a cluster. The CTAs of a cluster are packed onto as few SMs as hold them, so a launch that would fill the
// GPU with one or two CTAs per SM leaves half of it idle at four. From nine tokens on the launch therefore asks for as much
// shared memory as makes it spread: as few CTAs per SM as still hold all of it at once. (us a call in a chain of them,
// without and with: 28672 in blocks of 128 at 16, 24, 39 tokens 4.2, 4.9, 5.8 and 3.5, 4.2, 5.2; 14336 in blocks of 2048 at 64
// and 100 7.2, 8.4 and 5.3, 7.2. More tokens than fit at three per SM are faster packed: 200 of those 12.1 and 12.9; eight
// and fewer do not notice.)
template <int C>
int launch_quantize_cluster(const rcp::QuantParams& qp, int M, int T, size_t smem, cudaStream_t st) {
  static std::mutex mu;
  static bool attr_set[kMaxDevices] = {};
  static int fit[kMaxDevices][4] = {};   // clusters resident at once with r CTAs per SM
  auto kern = rcp::quantize_act_kernel<C>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)M * C);
  cfg.blockDim = dim3(T);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  if (C > 1 && M > 8) {
    RCP_CUDA(set_max_smem(kern, (int)smem_for_residency(1), mu, attr_set));
    int dev = 0;
    RCP_CUDA(cudaGetDevice(&dev));   // (below kMaxDevices: set_max_smem has looked)
    for (int r = 1; r <= 3 && (r + 1) * T <= 2048; r++) {   // (by its threads an SM takes no more than that anyway)
      std::lock_guard<std::mutex> lock(mu);
      if (!fit[dev][r]) {
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        cfg.dynamicSmemBytes = smem_for_residency(r);
        RCP_CUDA(cudaOccupancyMaxActiveClusters(&fit[dev][r], kern, &cfg));
      }
      if (M <= fit[dev][r]) {
        smem = std::max(smem, smem_for_residency(r));
        break;
      }
    }
  }
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = C > 1 ? attr : attr + 1;
  cfg.numAttrs = C > 1 ? 2 : 1;
  RCP_CUDA(cudaLaunchKernelEx(&cfg, kern, qp));
  return RCP_OK;
}

template <bool GRP, bool SDBG, bool HALF = false>
int launch_w3(const rcp::W3Params& wp, size_t smem, cudaStream_t st) {
  static std::mutex mu;
  static bool attr_set[kMaxDevices] = {};
  auto kern = rcp::gemv_w3a4_kernel<GRP, SDBG, HALF>;
  RCP_CUDA(set_max_smem(kern, rcp::kMaxK + 128, mu, attr_set));
  // One wave of resident CTAs, rows dealt round-robin to their warps (measured: CTAs beyond the resident wave,
  // and warps sharing a row along K, both cost more than the evener load returns). How many that is depends on the kernel
  // and on smem, a multiple of 4096 bytes up to kMaxK: asked once for each.
  static int resident[kMaxDevices][rcp::kMaxK / 4096 + 1] = {};
  int dev = 0, per_sm = 0;
  RCP_CUDA(cudaGetDevice(&dev));   // (below kMaxDevices: set_max_smem has looked)
  {
    std::lock_guard<std::mutex> lock(mu);
    int& known = resident[dev][smem / 4096];
    if (!known) {
      RCP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&known, kern, rcp::kW3Threads, smem));
      known = std::max(known, 1);
    }
    per_sm = known;
  }
  const int warps_per_cta = rcp::kW3Threads / 32;
  const int grid = std::min(sm_count() * per_sm, (wp.N + warps_per_cta - 1) / warps_per_cta);
  RCP_CUDA(launch_overlapped(kern, dim3(grid), dim3(rcp::kW3Threads), smem, st, wp));
  return RCP_OK;
}

}  // namespace

extern "C" {

const char* rcp_status_str(int status) {
  switch (status) {
    case RCP_OK: return "ok";
    case RCP_ERR_NULL: return "null pointer";
    case RCP_ERR_SHAPE: return "unsupported shape";
    case RCP_ERR_ALIGN: return "pointer not 16-byte aligned";
    case RCP_ERR_CODE: return "weight code above 3";
    case RCP_ERR_WORKSPACE: return "workspace missing";
    case RCP_ERR_CUDA: return "CUDA error";
    case RCP_ERR_VARIANT: return "kernel variant unknown or not applicable to this shape";
    case RCP_ERR_LIMIT: return "size beyond the entry point's fixed capacity";
    default: return "unknown status";
  }
}

int rcp_last_cuda_error(void) { return g_last_cuda_error; }

#ifndef RCP_HEADER_ID
#define RCP_HEADER_ID 0ull
#endif
unsigned long long rcp_header_id(void) { return RCP_HEADER_ID; }

int rcp_pack_weights(const uint8_t* codes, int N, int K, uint32_t* words, void* stream) {
  if (!codes || !words) return RCP_ERR_NULL;
  if (N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (!aligned16(codes) || !aligned16(words)) return RCP_ERR_ALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int* bad = nullptr;
  RCP_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&bad), g_pack_bad));
  bad += g_pack_next.fetch_add(1) % kPackSlots;
  RCP_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), st));
  const size_t nwords = (size_t)N * (K / 16);
  const int block = 256;
  const int grid = (int)std::min<size_t>((nwords + block - 1) / block, (size_t)148 * 32);
  rcp::pack_weights_kernel<<<grid, block, 0, st>>>(reinterpret_cast<const uint4*>(codes), nwords, words, bad);
  RCP_CUDA(cudaGetLastError());
  int h_bad = 0;
  RCP_CUDA(cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  RCP_CUDA(cudaStreamSynchronize(st));
  return h_bad ? RCP_ERR_CODE : RCP_OK;
}

int rcp_pack_weights3(const uint8_t* codes, int N, int K, uint32_t* words2, uint32_t* words1, void* stream) {
  if (!codes || !words2 || !words1) return RCP_ERR_NULL;
  if (N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (!aligned16(codes) || !aligned16(words2) || !aligned16(words1)) return RCP_ERR_ALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  int* bad = nullptr;
  RCP_CUDA(cudaGetSymbolAddress(reinterpret_cast<void**>(&bad), g_pack_bad));
  bad += g_pack_next.fetch_add(1) % kPackSlots;
  RCP_CUDA(cudaMemsetAsync(bad, 0, sizeof(int), st));
  const size_t nplane = (size_t)N * (K / 32);
  const int block = 256;
  const int grid = (int)std::min<size_t>((nplane + block - 1) / block, (size_t)sm_count() * 32);
  rcp::pack_weights3_kernel<<<grid, block, 0, st>>>(reinterpret_cast<const uint4*>(codes), nplane, words2, words1, bad);
  RCP_CUDA(cudaGetLastError());
  int h_bad = 0;
  RCP_CUDA(cudaMemcpyAsync(&h_bad, bad, sizeof(int), cudaMemcpyDeviceToHost, st));
  RCP_CUDA(cudaStreamSynchronize(st));
  return h_bad ? RCP_ERR_CODE : RCP_OK;
}

int rcp_gemv_w3a4(const uint32_t* words2, const uint32_t* words1, const void* lut_f16, int group, const uint8_t* xq,
                  const void* scale_f16, int M, int N, int K, void* y_f16, int32_t* S_dbg, void* stream) {
  if (!words2 || !words1 || !lut_f16 || !xq || !scale_f16 || !y_f16) return RCP_ERR_NULL;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (group != 0 && (group != 128 || K % 128)) return RCP_ERR_SHAPE;
  if (!aligned16(words2) || !aligned16(words1) || !aligned16(lut_f16) || !aligned16(xq) || !aligned16(S_dbg) ||
      (reinterpret_cast<uintptr_t>(y_f16) & 1u) || (reinterpret_cast<uintptr_t>(scale_f16) & 1u))
    return RCP_ERR_ALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // The last lane step of a row (64 units of 64 codes) is at most half full, and the row has so few steps that leaving half of
  // one out returns more than the 8 % that the form costs by its spills (4096x14336, an eighth of four steps: 15.1 -> 13.9 us)
  const bool half = (K / 64 - 1) % 64 < 32 && K <= 5 * 4096;
  const int ngrp = group ? K / 128 : 1;
  const size_t smem = (size_t)((K / 64 + 63) / 64) * 4096;   // expanded activations, K padded to whole lane steps of 4096 codes
  for (int m = 0; m < M; m++) {   // one token per launch: the variant is tuned for decoding one token
    rcp::W3Params wp;
    wp.words2 = words2; wp.words1 = words1;
    wp.lut = static_cast<const uint4*>(lut_f16);
    wp.xq = xq + (size_t)m * (K / 2);
    wp.scale = static_cast<const __half*>(scale_f16) + m;
    wp.y = static_cast<__half*>(y_f16) + (size_t)m * N;
    wp.S_out = S_dbg ? S_dbg + (size_t)m * N * ngrp * 8 : nullptr;
    wp.N = N; wp.K = K;
    int rc;
    if (group) rc = S_dbg ? launch_w3<true, true>(wp, smem, st) : launch_w3<true, false>(wp, smem, st);
    else if (half) rc = S_dbg ? launch_w3<false, true, true>(wp, smem, st) : launch_w3<false, false, true>(wp, smem, st);
    else rc = S_dbg ? launch_w3<false, true>(wp, smem, st) : launch_w3<false, false>(wp, smem, st);
    if (rc != RCP_OK) return rc;
  }
  return RCP_OK;
}

int rcp_nf3_export(const void* w_f16, const float* sig_beta, const float* sig_gamma, const float* sig_s1,
                   const float* table8_host, int zero_index, int N, int K, int group, uint32_t* words2,
                   uint32_t* words1, void* lut_f16, void* stream) {
  if (!w_f16 || !sig_beta || !sig_gamma || !sig_s1 || !table8_host || !words2 || !words1 || !lut_f16) return RCP_ERR_NULL;
  if (N < 1 || !k_ok(K) || group < 32 || group % 32 || K % group) return RCP_ERR_SHAPE;
  if (zero_index < 0 || zero_index > 7 || table8_host[zero_index] != 0.0f) return RCP_ERR_SHAPE;
  for (int i = 1; i < 8; i++)
    if (!(table8_host[i] > table8_host[i - 1])) return RCP_ERR_SHAPE;   // ascending (and no NaN)
  if (!aligned16(w_f16) || !aligned16(words2) || !aligned16(words1) || !aligned16(lut_f16) ||
      (reinterpret_cast<uintptr_t>(sig_beta) & 3u) || (reinterpret_cast<uintptr_t>(sig_gamma) & 3u) ||
      (reinterpret_cast<uintptr_t>(sig_s1) & 3u))
    return RCP_ERR_ALIGN;
  rcp::Nf3Params np;
  np.w = static_cast<const __half*>(w_f16);
  np.sb = sig_beta; np.sg = sig_gamma; np.s1 = sig_s1;
  np.words2 = words2; np.words1 = words1;
  np.lut = static_cast<uint4*>(lut_f16);
  for (int i = 0; i < 8; i++) np.table[i] = table8_host[i];
  np.zero = zero_index;
  np.N = N; np.K = K; np.G = group;
  np.units = (long long)N * (K / group);
  const int block = 256;
  const long long want = (np.units + (block / 32) - 1) / (block / 32);
  const int grid = (int)std::min<long long>(want, (long long)sm_count() * 16);
  rcp::nf3_export_kernel<<<grid, block, 0, static_cast<cudaStream_t>(stream)>>>(np);
  RCP_CUDA(cudaGetLastError());
  return RCP_OK;
}

int rcp_ldp_export(const void* w_f16, const float* sig_beta, const float* sig_gamma, const float* sig_s1,
                   const float* sig_s2, int N, int K, int group, uint32_t* words, void* lut_f16, void* stream) {
  if (!w_f16 || !sig_beta || !sig_gamma || !sig_s1 || !sig_s2 || !words || !lut_f16) return RCP_ERR_NULL;
  if (N < 1 || !k_ok(K) || group < 16 || group % 16 || K % group) return RCP_ERR_SHAPE;
  if (!aligned16(w_f16) || !aligned16(words) || (reinterpret_cast<uintptr_t>(lut_f16) & 7u) ||
      (reinterpret_cast<uintptr_t>(sig_beta) & 3u) || (reinterpret_cast<uintptr_t>(sig_gamma) & 3u) ||
      (reinterpret_cast<uintptr_t>(sig_s1) & 3u) || (reinterpret_cast<uintptr_t>(sig_s2) & 3u))
    return RCP_ERR_ALIGN;
  rcp::LdpParams lp;
  lp.w = static_cast<const __half*>(w_f16);
  lp.sb = sig_beta; lp.sg = sig_gamma; lp.s1 = sig_s1; lp.s2 = sig_s2;
  lp.words = words;
  lp.lut = static_cast<uint2*>(lut_f16);
  lp.N = N; lp.K = K; lp.G = group;
  lp.units = (long long)N * (K / group);
  const int block = 256;
  // From 4096 units on a warp takes tiles of 32 of them. Fewer are too few tiles for the GPU, and a tile is 32 units worked on
  // one after the other: there a warp per unit is faster (us, a warp per unit against tiles: 64 units 2.7 and 3.1, 512 2.9
  // and 3.9, 2048 3.1 and 3.9, 4096 3.9 and 3.9, 8192 6.0 and 4.0).
  if (group == rcp::kLdpGroup && lp.units >= 4096) {
    static std::mutex mu;
    static bool attr_set[kMaxDevices] = {};
    RCP_CUDA(set_max_smem(rcp::ldp_export128_kernel, (int)rcp::kLdpSmem, mu, attr_set));
    const long long tiles = (lp.units + 31) / 32;   // a warp per 32 units, two CTAs per SM
    const int g128 = (int)std::min<long long>((tiles + rcp::kLdpWarps - 1) / rcp::kLdpWarps, 2 * sm_count());
    rcp::ldp_export128_kernel<<<g128, rcp::kLdpWarps * 32, rcp::kLdpSmem, static_cast<cudaStream_t>(stream)>>>(lp);
    RCP_CUDA(cudaGetLastError());
    return RCP_OK;
  }
  const long long want = (lp.units + (block / 32) - 1) / (block / 32);
  const int grid = (int)std::min<long long>(want, (long long)sm_count() * 16);
  rcp::ldp_export_kernel<<<grid, block, 0, static_cast<cudaStream_t>(stream)>>>(lp);
  RCP_CUDA(cudaGetLastError());
  return RCP_OK;
}

int rcp_quantize_act(const void* x_f16, int M, int K, int had_block, float clip_ratio, uint8_t* xq,
                     void* scale_f16, void* stream) {
  if (!x_f16 || !xq || !scale_f16) return RCP_ERR_NULL;
  if (M < 1 || M > 65535 || !k_ok(K)) return RCP_ERR_SHAPE;
  int B = had_block <= 1 ? 1 : had_block;
  if (B > 8192 || (B & (B - 1)) || K % B) return RCP_ERR_SHAPE;
  if (!(clip_ratio > 0.f) || !std::isfinite(clip_ratio)) return RCP_ERR_SHAPE;
  if (!aligned16(x_f16) || !aligned16(xq) || (reinterpret_cast<uintptr_t>(scale_f16) & 1u)) return RCP_ERR_ALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);

  // A cluster of C CTAs per token, 8 elements per thread, about 2048 elements per CTA (8192 at most).
  rcp::QuantParams qp;
  qp.x = static_cast<const __half*>(x_f16);
  qp.xq = xq;
  qp.scale = static_cast<__half*>(scale_f16);
  qp.K = K; qp.B = B;
  qp.lgB = 0;
  while ((1 << qp.lgB) < B) qp.lgB++;
  qp.inv_sqrt_b = (float)(1.0 / std::sqrt((double)B));
  qp.clip_ratio = std::min(clip_ratio, rcp::kClipRatioCap);
  if (rows_form(M, K, B)) return launch_quantize_rows(qp, M, st);
  // whole rotation blocks per CTA
  int C = 1;
  while (C < 8 && K / (2 * C) >= 2048) C *= 2;
  qp.unit = std::max(B, 64);
  qp.nunits = K / qp.unit;
  qp.lg_local = qp.lgB;
  C = std::min(C, qp.nunits);
  while (C > 1 && (C & (C - 1))) C--;   // power of two
  int per = (qp.nunits + C - 1) / C;
  while ((long long)per * qp.unit > 8192 && C < 8) { C *= 2; per = (qp.nunits + C - 1) / C; }
  if ((long long)per * qp.unit > 8192) return RCP_ERR_SHAPE;
  const int T = (per * qp.unit / 8 + 31) / 32 * 32;
  const size_t smem = B > 256 ? (size_t)T * 8 * sizeof(float) : 0;
  switch (C) {
    case 1: return launch_quantize_cluster<1>(qp, M, T, smem, st);
    case 2: return launch_quantize_cluster<2>(qp, M, T, smem, st);
    case 4: return launch_quantize_cluster<4>(qp, M, T, smem, st);
    default: return launch_quantize_cluster<8>(qp, M, T, smem, st);
  }
}

int rcp_gemv_plan(int M, int N, int K, int sms, int* out, int cap) {
  if (!out && cap > 0) return RCP_ERR_NULL;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (sms <= 0) sms = 148;
  int nsplit = 1;
  const int mp = tokens_and_parts(M, N, K, 16, sms, &nsplit);
  const StreamPlan pl = make_plan(mp, N, K, sms, false, 0, nsplit);
  int v[7 + 5 * rcp::kMaxPhases];
  int n = 0;
  v[n++] = mp;
  v[n++] = (M + mp - 1) / mp;
  v[n++] = pl.stages;
  v[n++] = (int)pl.smem;
  v[n++] = pl.nchunk;
  v[n++] = pl.nphase;
  for (int i = 0; i < pl.nphase; i++) {
    v[n++] = pl.phase[i].gpc; v[n++] = pl.phase[i].first; v[n++] = pl.phase[i].total;
    v[n++] = pl.phase[i].ncta; v[n++] = pl.phase[i].reps;
  }
  v[n++] = pl.nsplit;
  for (int i = 0; i < n && i < cap; i++) out[i] = v[i];
  return n;
}

int rcp_gemv_umma_plan(int M, int N, int K, int sms, int had_block, int* out, int cap) {
  if (!out && cap > 0) return RCP_ERR_NULL;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (sms <= 0) sms = 148;
  if (had_block != 0 && !fused_ok(M, K, had_block)) return RCP_ERR_VARIANT;
  UmmaChoice c;
  umma_choose(M, N, K, sms, had_block != 0 && full_block(K, had_block) ? rcp::full_rotate_bytes(K) : 0, c);
  int n = 0;
  auto put = [&](long long v) { if (n < cap) out[n] = (int)v; n++; };
  put(c.faster + 2 * c.faster_late);
  put(c.launches);
  for (int i = 0; i < c.launches; i++) {
    const UmmaPlan& pl = i + 1 < c.launches ? c.plan : c.last;
    for (const long long v : {(long long)std::min(c.tokens, M - i * c.tokens), (long long)pl.tokens, (long long)pl.stages, (long long)pl.smem,
                              (long long)pl.nchunk, (long long)pl.part_chunks, (long long)pl.kpl, (long long)pl.bhalf, (long long)pl.bstep,
                              (long long)pl.bgroup, (long long)pl.lg_m2, (long long)pl.slots, (long long)pl.dcols, (long long)pl.acc_cols, (long long)pl.nbuf,
                              (long long)pl.helpers, (long long)pl.off_bar, (long long)pl.off_misc, (long long)pl.off_red, (long long)pl.red_bytes,
                              (long long)pl.off_bs, (long long)pl.bs_bytes, (long long)pl.off_qbuf, (long long)pl.nphase})
      put(v);
    for (int j = 0; j < pl.nphase; j++) {
      const rcp::UmmaPhase& ph = pl.phase[j];
      for (const int v : {ph.gpc, ph.first, ph.total, ph.ncta, ph.reps, ph.kp, ph.items, ph.ncol, ph.ncol_f8}) put(v);
    }
  }
  return n;
}

size_t rcp_gemv_workspace_bytes(int M, int N, int K) {
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return 0;
  return 16;   // a status word for the kernels' bounded waits; no sums pass through global memory
}

// The kernel for a call, as measured on B200: umma_faster; otherwise one token runs fastest on the CUDA cores, more tokens on mma.sync.
static int auto_variant(int M, int N, int K, bool late_start) {
  const UmmaChoice& c = umma_choice(M, N, K, 0);
  return (late_start ? c.faster_late : c.faster) ? RCP_GEMV_UMMA : M == 1 ? RCP_GEMV_DP4A : RCP_GEMV_MMA_ONLY;
}

// late_start: the call quantizes its activations itself (see the end of gemv_stream_kernel)
static int gemv_w2a4(int variant, const uint32_t* words, const void* lut_f16, const uint8_t* xq, const void* scale_f16, int M,
                     int N, int K, void* y_f16, void* workspace, int32_t* S_dbg, void* stream, bool late_start) {
  if (!words || !lut_f16 || !xq || !scale_f16 || !y_f16) return RCP_ERR_NULL;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (!aligned16(words) || !aligned16(xq) || !aligned16(S_dbg) ||
      (reinterpret_cast<uintptr_t>(lut_f16) & 7u) || (reinterpret_cast<uintptr_t>(y_f16) & 1u) ||
      (reinterpret_cast<uintptr_t>(scale_f16) & 1u))
    return RCP_ERR_ALIGN;
  if (reinterpret_cast<uintptr_t>(workspace) & 3u) return RCP_ERR_ALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // S_dbg without a variant of the caller's choice: the plain kernel. With one: the checked instantiation of
  // that streaming kernel, which stores the sums it finishes its rows from.
  if (S_dbg && variant == RCP_GEMV_AUTO) variant = RCP_GEMV_SIMPLE;
  if (variant == RCP_GEMV_AUTO) variant = auto_variant(M, N, K, late_start);
  // the streaming kernels wait on barriers with a bound and report a wait that gave up through the workspace
  if (variant != RCP_GEMV_SIMPLE && !workspace) return RCP_ERR_WORKSPACE;
  switch (variant) {
    case RCP_GEMV_SIMPLE: {
      const int block = 256;
      const int grid = (N + (block / 32) - 1) / (block / 32);
      rcp::gemv_simple_kernel<<<grid, block, 0, st>>>(words, static_cast<const uint2*>(lut_f16), xq,
                                                      static_cast<const __half*>(scale_f16), M, N, K,
                                                      static_cast<__half*>(y_f16), S_dbg);
      break;
    }
    case RCP_GEMV_MMA:
      // tensor-core path; for one or two tokens the b0*b1 plane goes to dp4a (FMA pipe) instead
      return launch_stream_passes(M <= 2 ? rcp::kModeHybrid : rcp::kModeMma, 16, words, lut_f16, xq, scale_f16, M, N, K,
                                  y_f16, workspace, st, false, S_dbg, late_start);
    case RCP_GEMV_MMA_ONLY:
      return launch_stream_passes(rcp::kModeMma, 16, words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace, st, false,
                                  S_dbg, late_start);
    case RCP_GEMV_DP4A:
      // CUDA-core path: two tokens per launch
      return launch_stream_passes(rcp::kModeDp4a, 2, words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace, st, false,
                                  S_dbg);
    case RCP_GEMV_UMMA:
      return launch_umma_passes(words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace, st, S_dbg, late_start);
    case RCP_GEMV_MMA_STREAM: {
      // tensor-core path with the activations streamed beside the weights: all tokens in one launch, any K
      const StreamPlan pl = make_plan(M, N, K, sm_count(), false, 0, 1, true);
      if (pl.stages < 2 || pl.smem > kSmemMax) return RCP_ERR_VARIANT;
      return launch_stream(rcp::kModeMma, words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace, st, false, nullptr,
                           nullptr, 1, nullptr, S_dbg, true, late_start);
    }
    default:
      return RCP_ERR_VARIANT;
  }
  RCP_CUDA(cudaGetLastError());
  return RCP_OK;
}

int rcp_gemv_w2a4_variant(int variant, const uint32_t* words, const void* lut_f16, const uint8_t* xq,
                          const void* scale_f16, int M, int N, int K, void* y_f16, void* workspace,
                          int32_t* S_dbg, void* stream) {
  return gemv_w2a4(variant, words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace, S_dbg, stream, false);
}

int rcp_gemv_w2a4(const uint32_t* words, const void* lut_f16, const uint8_t* xq, const void* scale_f16,
                  int M, int N, int K, void* y_f16, void* workspace, int32_t* S_dbg, void* stream) {
  return rcp_gemv_w2a4_variant(RCP_GEMV_AUTO, words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace,
                               S_dbg, stream);
}

int rcp_gemv_w2a16_checked(const uint32_t* words, const void* lut_f16, const void* x_f16, int M, int N, int K,
                           void* y_f16, int8_t* digits, float* unit, void* workspace, int32_t* S_dbg, void* stream) {
  if (!words || !lut_f16 || !x_f16 || !y_f16 || !digits || !unit) return RCP_ERR_NULL;
  if (!workspace) return RCP_ERR_WORKSPACE;
  if (!aligned16(S_dbg)) return RCP_ERR_ALIGN;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (!aligned16(words) || !aligned16(x_f16) || !aligned16(digits) || (reinterpret_cast<uintptr_t>(lut_f16) & 7u) ||
      (reinterpret_cast<uintptr_t>(y_f16) & 1u) || (reinterpret_cast<uintptr_t>(unit) & 3u) ||
      (reinterpret_cast<uintptr_t>(workspace) & 3u))
    return RCP_ERR_ALIGN;
  // digit columns per launch: sixteen (four tokens) or eight (two) where their expanded bytes fit, else four
  const int cols = 4 * M;
  int nsplit = 1;
  const int cp = tokens_and_parts(std::min(cols, 16), N, K, 16, sm_count(), &nsplit) & ~3;
  if (cp < 4) return RCP_ERR_SHAPE;   // not even the four digit planes of one token fit (very many rows and a long K)
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // One token of up to 16384 elements: one kernel does both steps (every CTA splits its own copy of the
  // activations, held in registers between the search for the largest magnitude and the digits, which costs
  // less than a launch in front of it: measured 0.4 to 1.2 us a call; with two tokens the launch in front won).
  if (M == 1 && nsplit == 1 && cp == cols && K <= 16384 &&
      make_plan(cols, N, K, sm_count(), false, (size_t)cols * K, 1).stages >= 3) {
    const SplitAct sa{x_f16, digits, unit};
    return launch_stream(rcp::kModeMma, words, lut_f16, nullptr, nullptr, cols, N, K, y_f16, workspace, st, false,
                         nullptr, nullptr, 1, &sa, S_dbg);
  }
  // half of the threads have a vector of eight elements (a whole one each: 0.1 to 0.4 us a call slower)
  const int parts = std::max(1, std::min(16, K / (4 * rcp::kSplitThreads)));
  RCP_CUDA(launch_overlapped(rcp::split_act16_kernel, dim3(M * parts), dim3(rcp::kSplitThreads), 0, st,
                             static_cast<const __half*>(x_f16), K, parts, digits, unit));
  for (int c0 = 0; c0 < cols; c0 += cp) {
    const int cc = std::min(cp, cols - c0);
    const int rc = launch_stream(rcp::kModeMma, words, lut_f16, reinterpret_cast<const uint8_t*>(digits) + (size_t)c0 * K,
                                 nullptr, cc, N, K, static_cast<__half*>(y_f16) + (size_t)(c0 / 4) * N, workspace, st,
                                 false, nullptr, unit + c0, nsplit, nullptr, S_dbg ? S_dbg + (size_t)c0 * N * 4 : nullptr, false, true);
    if (rc != RCP_OK) return rc;
  }
  return RCP_OK;
}

int rcp_gemv_w2a16(const uint32_t* words, const void* lut_f16, const void* x_f16, int M, int N, int K, void* y_f16,
                   int8_t* digits, float* unit, void* workspace, void* stream) {
  return rcp_gemv_w2a16_checked(words, lut_f16, x_f16, M, N, K, y_f16, digits, unit, workspace, nullptr, stream);
}

static int gemv_w2a4_grouped(int variant, const uint32_t* words, const void* lut_f16, int group, const uint8_t* xq,
                             const void* scale_f16, int M, int N, int K, void* y_f16, void* workspace, int32_t* S_dbg,
                             void* stream, bool late_start) {
  if (!words || !lut_f16 || !xq || !scale_f16 || !y_f16) return RCP_ERR_NULL;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (group < 16 || group % 16 || K % group) return RCP_ERR_SHAPE;
  if (!aligned16(words) || !aligned16(xq) || !aligned16(S_dbg) ||
      (reinterpret_cast<uintptr_t>(lut_f16) & 7u) || (reinterpret_cast<uintptr_t>(y_f16) & 1u) ||
      (reinterpret_cast<uintptr_t>(scale_f16) & 1u))
    return RCP_ERR_ALIGN;
  if (reinterpret_cast<uintptr_t>(workspace) & 3u) return RCP_ERR_ALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // the streaming kernels are built for the paper's group size; other sizes take the plain kernel
  if (variant == RCP_GEMV_AUTO && (S_dbg || group != 128)) variant = RCP_GEMV_SIMPLE;
  if (variant == RCP_GEMV_AUTO) variant = (M <= 2) ? RCP_GEMV_DP4A : RCP_GEMV_MMA_ONLY;
  if (variant != RCP_GEMV_SIMPLE && !workspace) return RCP_ERR_WORKSPACE;
  switch (variant) {
    case RCP_GEMV_SIMPLE: {
      const int block = 256;
      const int grid = (N + (block / 32) - 1) / (block / 32);
      rcp::gemv_simple_grouped_kernel<<<grid, block, 0, st>>>(words, static_cast<const uint2*>(lut_f16), xq,
                                                              static_cast<const __half*>(scale_f16), M, N, K, group,
                                                              static_cast<__half*>(y_f16), S_dbg);
      break;
    }
    case RCP_GEMV_MMA_ONLY:
      if (group != 128) return RCP_ERR_VARIANT;
      return launch_stream_passes(rcp::kModeMma, 8, words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace, st, true,
                                  S_dbg, late_start);
    case RCP_GEMV_DP4A:
      if (group != 128) return RCP_ERR_VARIANT;
      return launch_stream_passes(rcp::kModeDp4a, 2, words, lut_f16, xq, scale_f16, M, N, K, y_f16, workspace, st, true,
                                  S_dbg);
    default:
      return RCP_ERR_VARIANT;
  }
  RCP_CUDA(cudaGetLastError());
  return RCP_OK;
}

int rcp_gemv_w2a4_grouped_variant(int variant, const uint32_t* words, const void* lut_f16, int group,
                                  const uint8_t* xq, const void* scale_f16, int M, int N, int K, void* y_f16,
                                  void* workspace, int32_t* S_dbg, void* stream) {
  return gemv_w2a4_grouped(variant, words, lut_f16, group, xq, scale_f16, M, N, K, y_f16, workspace, S_dbg, stream, false);
}

int rcp_gemv_w2a4_grouped(const uint32_t* words, const void* lut_f16, int group, const uint8_t* xq,
                          const void* scale_f16, int M, int N, int K, void* y_f16, void* workspace, int32_t* S_dbg,
                          void* stream) {
  return rcp_gemv_w2a4_grouped_variant(RCP_GEMV_AUTO, words, lut_f16, group, xq, scale_f16, M, N, K, y_f16, workspace,
                                       S_dbg, stream);
}

int rcp_gemv_w2a4_static(const uint32_t* words, const void* lut_f16, const uint8_t* xq, const void* scale_f16,
                         int M, int N, int K, void* y_f16, void* stream) {
  // the same checks as rcp_gemv_w2a4, before anything is put on the stream
  if (!words || !lut_f16 || !xq || !scale_f16 || !y_f16) return RCP_ERR_NULL;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  if (!aligned16(words) || !aligned16(xq) || (reinterpret_cast<uintptr_t>(lut_f16) & 7u) ||
      (reinterpret_cast<uintptr_t>(y_f16) & 1u) || (reinterpret_cast<uintptr_t>(scale_f16) & 1u))
    return RCP_ERR_ALIGN;
  const size_t need = rcp_gemv_workspace_bytes(M, N, K);
  if (need > RCP_STATIC_SCRATCH_BYTES) return RCP_ERR_LIMIT;
  void* scratch = nullptr;
  const int rc = static_scratch_address(&scratch);
  if (rc != RCP_OK) return rc;
  // the array keeps the previous call's contents: clear what this call's kernel expects to be zero
  if (need > 0) RCP_CUDA(cudaMemsetAsync(scratch, 0, need, static_cast<cudaStream_t>(stream)));
  return rcp_gemv_w2a4_variant(RCP_GEMV_AUTO, words, lut_f16, xq, scale_f16, M, N, K, y_f16, scratch, nullptr,
                               stream);
}

int rcp_gemv_w2a4_static_status(int32_t* status_host, void* stream) {
  if (!status_host) return RCP_ERR_NULL;
  void* scratch = nullptr;
  const int rc = static_scratch_address(&scratch);
  if (rc != RCP_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  RCP_CUDA(cudaMemcpyAsync(status_host, scratch, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  RCP_CUDA(cudaStreamSynchronize(st));
  return RCP_OK;
}

int rcp_selftest_wait_timeout(void* workspace, int polls, void* stream) {
  if (polls < 1 || polls > (1 << 20)) return RCP_ERR_SHAPE;
  if (reinterpret_cast<uintptr_t>(workspace) & 3u) return RCP_ERR_ALIGN;
  void* status = workspace;
  if (!status) {
    const int rc = static_scratch_address(&status);
    if (rc != RCP_OK) return rc;
  }
  rcp::wait_timeout_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(static_cast<int32_t*>(status), (uint32_t)polls);
  RCP_CUDA(cudaGetLastError());
  return RCP_OK;
}

int rcp_linear_w2a4_launches(int M, int N, int K, int had_block, int group) {
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  const int B = had_block <= 1 ? 1 : had_block;
  if (fused_ok(M, K, B) && (group == 0 || group == 128)) return 1;
  if (group != 0 && group != 128) return 2;
  const int cap = group == 0 ? (M == 1 ? 2 : 16) : (M <= 2 ? 2 : 8);   // tokens per launch of the variant AUTO picks
  int nsplit = 1;
  if (group == 0 && umma_choice(M, N, K, 0).faster_late) return 1 + umma_choice(M, N, K, 0).launches;
  const int mp = (group != 0 || cap < 8) ? tokens_per_pass(M, K, cap) : tokens_and_parts(M, N, K, cap, sm_count(), &nsplit);
  return 1 + (M + mp - 1) / mp;
}

int rcp_linear_w2a4_checked(const void* x_f16, int M, int K, int had_block, float clip_ratio, const uint32_t* words,
                            const void* lut_f16, int group, int N, void* y_f16, uint8_t* xq, void* scale_f16,
                            void* workspace, int32_t* S_dbg, void* stream) {
  if (!x_f16 || !words || !lut_f16 || !y_f16) return RCP_ERR_NULL;
  if (!aligned16(S_dbg)) return RCP_ERR_ALIGN;
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  const int B = had_block <= 1 ? 1 : had_block;
  if (B > 8192 || (B & (B - 1)) || K % B) return RCP_ERR_SHAPE;
  if (!(clip_ratio > 0.f) || !std::isfinite(clip_ratio)) return RCP_ERR_SHAPE;
  if (group != 0 && (group < 16 || group % 16 || K % group)) return RCP_ERR_SHAPE;
  if (!aligned16(x_f16) || !aligned16(words) || !aligned16(xq) || (reinterpret_cast<uintptr_t>(lut_f16) & 7u) ||
      (reinterpret_cast<uintptr_t>(y_f16) & 1u) || (reinterpret_cast<uintptr_t>(scale_f16) & 1u) ||
      (reinterpret_cast<uintptr_t>(workspace) & 3u))
    return RCP_ERR_ALIGN;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (!workspace) return RCP_ERR_WORKSPACE;
  if (!(M == 1 && B == K && (K == 4096 || K == 8192)) && (!xq || !scale_f16)) return RCP_ERR_NULL;
  if (fused_ok(M, K, B) && (group == 0 || group == 128)) {
    const FusedAct fa{x_f16, B, clip_ratio, xq, scale_f16};
    if (group == 0) {
      const UmmaChoice& c = umma_choice(M, N, K, full_block(K, B) ? rcp::full_rotate_bytes(K) : 0);
      if (c.faster) return launch_umma(words, lut_f16, nullptr, nullptr, M, N, K, y_f16, workspace, st, c.plan, &fa, S_dbg, false);
    }
    return launch_stream(rcp::kModeDp4a, words, lut_f16, nullptr, nullptr, M, N, K, y_f16, workspace, st, group == 128,
                         &fa, nullptr, 1, nullptr, S_dbg);
  }
  // otherwise the two kernels one after the other; they need the staging buffers
  if (!xq || !scale_f16) return RCP_ERR_NULL;
  int rc = rcp_quantize_act(x_f16, M, K, had_block, clip_ratio, xq, scale_f16, stream);
  if (rc != RCP_OK) return rc;
  // with S_dbg: the streaming kernel AUTO would pick, in its checked instantiation
  if (group == 0)
    return gemv_w2a4(S_dbg ? auto_variant(M, N, K, true) : RCP_GEMV_AUTO, words, lut_f16, xq, scale_f16, M,
                     N, K, y_f16, workspace, S_dbg, stream, true);
  return gemv_w2a4_grouped(S_dbg && group == 128 ? (M <= 2 ? RCP_GEMV_DP4A : RCP_GEMV_MMA_ONLY) : RCP_GEMV_AUTO, words,
                           lut_f16, group, xq, scale_f16, M, N, K, y_f16, workspace, S_dbg, stream, true);
}

int rcp_linear_w2a4(const void* x_f16, int M, int K, int had_block, float clip_ratio, const uint32_t* words,
                    const void* lut_f16, int group, int N, void* y_f16, uint8_t* xq, void* scale_f16, void* workspace,
                    void* stream) {
  return rcp_linear_w2a4_checked(x_f16, M, K, had_block, clip_ratio, words, lut_f16, group, N, y_f16, xq, scale_f16,
                                 workspace, nullptr, stream);
}

int rcp_linear_w2a4_host(const void* x_host_f16, int M, int K, int had_block, float clip_ratio,
                         const uint32_t* words, const void* lut_f16, int N, void* y_host_f16, void* x_dev,
                         uint8_t* xq_dev, void* scale_dev, void* y_dev, void* workspace, void* stream) {
  if (!x_host_f16 || !y_host_f16 || !x_dev || !y_dev) return RCP_ERR_NULL;   // staging is needed for pageable memory
  if (M < 1 || M > rcp::kMaxTokens || N < 1 || !k_ok(K)) return RCP_ERR_SHAPE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  // Page-locked host memory is visible to the GPU: the quantizer (a handful of CTAs) then reads the
  // few kilobytes of activations straight from it, which saves a trip through the copy engine. The
  // single-kernel form would have every CTA fetch them across the bus, so it is not used here.
  cudaPointerAttributes attr;
  const void* x_mapped = nullptr;
  if (xq_dev && scale_dev && cudaPointerGetAttributes(&attr, x_host_f16) == cudaSuccess &&
      attr.type == cudaMemoryTypeHost && attr.devicePointer && aligned16(attr.devicePointer))
    x_mapped = attr.devicePointer;
  else
    (void)cudaGetLastError();   // an unregistered pointer is not an error here
  // Likewise the GEMV can store its few kilobytes of results straight into page-locked host memory.
  void* y_mapped = nullptr;
  if (cudaPointerGetAttributes(&attr, y_host_f16) == cudaSuccess && attr.type == cudaMemoryTypeHost &&
      attr.devicePointer)
    y_mapped = attr.devicePointer;
  else
    (void)cudaGetLastError();
  void* const y_out = y_mapped ? y_mapped : y_dev;
  int rc;
  if (x_mapped) {
    rc = rcp_quantize_act(x_mapped, M, K, had_block, clip_ratio, xq_dev, scale_dev, stream);
    if (rc == RCP_OK)
      rc = gemv_w2a4(RCP_GEMV_AUTO, words, lut_f16, xq_dev, scale_dev, M, N, K, y_out, workspace, nullptr, stream, true);
  } else {
    RCP_CUDA(cudaMemcpyAsync(x_dev, x_host_f16, (size_t)M * K * 2, cudaMemcpyHostToDevice, st));
    rc = rcp_linear_w2a4(x_dev, M, K, had_block, clip_ratio, words, lut_f16, 0, N, y_out, xq_dev, scale_dev, workspace,
                         stream);
  }
  if (rc != RCP_OK) return rc;
  if (!y_mapped) RCP_CUDA(cudaMemcpyAsync(y_host_f16, y_dev, (size_t)M * N * 2, cudaMemcpyDeviceToHost, st));
  return RCP_OK;
}

}  // extern "C"
