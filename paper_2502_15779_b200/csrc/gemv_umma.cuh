// LUT GEMV on the fifth-generation tensor cores (Section 4.4 of the paper: O = S * X_q * LUT[W_q]).
//
// What an instruction costs. tcgen05.mma with its A operand in tensor memory takes 8 clocks for 128 rows x 32 bytes of A and up
// to 16 columns (16 clocks for 32, 64 for 128): 512 bytes of A per clock, where shared memory delivers 105. Columns are free,
// so a GEMV is as cheap here as a product with sixteen tokens, and the mask arithmetic that turns packed codes into A is
// what counts. (An issue loop whose operands the compiler cannot prove warp-uniform runs at 27 to 96 clocks an instruction,
// whatever its size.)
//
// Formulation. b0, b1: the bits of a code; per row and token T1 = sum b0 q, T2 = sum b1 q, T3 = sum b0 b1 q and T0 = sum q give
// the per-code sums S3 = T3, S1 = T1 - T3, S2 = T2 - T3, S0 = T0 - T1 - T2 + T3. A byte of a packed word holds four codes. Shifted
// so that one of them stands in bits 6 and 7 and masked there, a byte has the value
//   64 b0 + 128 b1 as an unsigned integer, 64 b0 - 128 b1 as a signed one, 2 b0 (1 - 2 b1) as an e4m3 number,
// three independent functions of the code: the same operand in tensor memory goes through three instructions (kind::i8
// with A unsigned, kind::i8 with A signed, kind::f8f6f4) and no product of bits is ever computed. Four masks and three
// shifts per 16 codes, where the CUDA-core kernel needs 23 operations and the mma.sync kernels 18 and 6 MMA slots.
// The activations are bytes 0..15, u = q + 8: as e4m3 such a byte is u / 512 (subnormals and the first binade are evenly
// spaced), so one copy serves all three instructions. A column of ones beside the tokens measures what the + 8 adds.
// The sums are exact: int32, and fp32 sums of multiples of 2^-8 below 2^13, 20 bits of 24. (That kind::f8f6f4 drops no bits below
// its largest product while it adds is measured, at the ends of the range too, not documented.)
//
// Work. Groups of 16 rows are shared out over the CTAs in phases like in gemv_stream.cuh; an item is 128 lanes x 128
// bytes of packed weights (16 KB): 16 gpc rows x kp chunks of K side by side in the lanes, each chunk with columns of its own
// (lane block j uses column block j, the other products are dropped). Warps: a producer streams the items' boxes into a ring
// (TMA, 128-byte swizzle); eight converters, two to a quarter of the lanes (a warp reads and writes the 32 lanes its number
// gives it), each half of an item's bytes, fill the slots of tensor memory with item after item; three issuers, one per
// reading; sixteen workers prepare the activations, then turn the sums of a tile into y while the next is worked on (four tokens
// to a warp; up to eight tokens the last eight of them convert too). Slots of 128 columns (a whole item): with 64 the handshakes
// cost 55 clocks per KB of weights, so 40, less than the 44 to 49 that HBM needs.
// What it measured (B200, us a call of the whole linear in a chain, cold weights; before: dp4a for one token, mma.sync for more):
// 57344x8192 at 1, 3, 8, 12, 16 tokens 30.5, 39.7, 38.8, 76.7, 75.7 -> 24.8, 28.1, 31.2, 33.5, 40.1; 28672x4096 at 16 23.7 -> 16.8;
// 8192x28672 at 8 31.3 -> 28.5. Bound: HBM in the loop up to eight tokens (an item per SM in 720 clocks is 6.4 TB/s; four times the
// weights, 28672x4096 at two tokens and 57344x8192 at one, take 14.2 us longer, 6.2 TB/s); at sixteen the 32 columns take 768 clocks
// an item; beside it some 5 us from launch to the first sums and from the last to y.
#pragma once
#include "gemv_stream.cuh"

namespace rcp {

constexpr int kUWork = 16;                              // workers: activations, then the tiles' ends
constexpr int kUConv = 8;                               // converters
constexpr int kUIssue = 3;
constexpr int kUFirstConv = kUWork, kUFirstIssue = kUFirstConv + kUConv, kUProducer = kUFirstIssue + kUIssue;
constexpr int kUThreads = (kUProducer + 1) * 32;
constexpr int kULanes = 128;
constexpr int kUItemBytes = kULanes * kChunkWords * 4;  // 16 KB
constexpr int kUMaxStages = 12;
constexpr int kUMaxSlots = 3, kUMaxBuf = 4;
constexpr int kUTok = 4;                                // tokens of a worker at a tile's end

struct UmmaPhase {
  int gpc, first, total, ncta, reps, q, r;   // as in GemvPhase
  int kp;      // chunks of K side by side in the lanes (a power of two; 16 gpc kp <= 128)
  int items;   // per repetition: ceil(nchunk / kp)
  int ncol;    // columns of the kind::i8 instructions: kp (M + 1), rounded up to 8 or a multiple of 16
  int ncol_f8; // of the e4m3 one: 16 at least
  int inv_rows;   // ceil(2^16 / (16 gpc)): v / (16 gpc) == (v * inv_rows) >> 16 for v < 512
};
struct UmmaParams {
  const uint2* lut;
  const uint8_t* xq;
  const __half* scale;
  __half* y;
  int32_t* status;
  int32_t* S_out;       // SDBG: [M][N][4]
  int M, N, K, nchunk, nphase;
  UmmaPhase phase[kMaxPhases];
  // quantizer inside (FQ), one token
  const __half* x;
  uint8_t* xq_out;
  __half* scale_out;
  float inv_sqrt_b, clip_ratio;
  int had_block;
  // activations in shared memory, strides in units of 16 bytes: 16-byte piece (chunk c, step s, position p, half h, row n)
  // at (c / kpl) bgroup + s bstep + (2 p + h) bhalf + (c % kpl)(M + 1) + n
  int kpl, lg_kpl, bgroup, bstep, bhalf;
  int part_chunks;      // chunks of K whose activations are in shared memory at a time (nchunk: all; else one tile per CTA at most)
  int helpers;          // the last eight workers have no tokens to finish: they become converters
  int lg_m2;            // log2 of M rounded up to a power of two
  // tensor memory: slots of 128 columns at the top, at the bottom nbuf sets of accumulators (acc_cols: dcols columns for each integer
  // reading, dcols or 16 for the e4m3 one behind them)
  int slots, dcols, acc_cols, nbuf;
  int stages, ramp_clk;
  int off_bar, off_misc, off_red, off_bs, off_qbuf;
  int red_bytes, bs_bytes;
};

__device__ __forceinline__ bool elect_one() {
  uint32_t pred;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xFFFFFFFF;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(pred));
  return pred != 0;
}
// Bounded wait of a whole warp. The vote makes the answer uniform for the compiler too: a loop that may be left lane by lane
// loses the uniform registers that tcgen05 instructions take their operands from.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < kSpinLimit; i++)
    if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
  return false;
}
__device__ __forceinline__ void tmem_st32(uint32_t at, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(at),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_ld1(uint32_t at, uint32_t& r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(at) : "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t at, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(at) : "memory");
}
// One instruction of a warp that stays together, issued by its lane with `elected` set (a branch around the instructions would
// take their operands out of the uniform registers). acc: whether the accumulators are added to or overwritten.
template <bool F8>
__device__ __forceinline__ void umma(uint32_t elected, uint32_t d, uint32_t a, uint32_t b_lo, uint32_t b_hi, uint32_t idesc, uint32_t acc) {
  if constexpr (F8)
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 bd;\n\tmov.b64 bd, {%2, %3};\n\tsetp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], bd, %4, p;\n\t}" ::"r"(d), "r"(a), "r"(b_lo), "r"(b_hi),
                 "r"(idesc), "r"(elected), "r"(acc) : "memory");
  else
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b64 bd;\n\tmov.b64 bd, {%2, %3};\n\tsetp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q tcgen05.mma.cta_group::1.kind::i8 [%0], [%1], bd, %4, p;\n\t}" ::"r"(d), "r"(a), "r"(b_lo), "r"(b_hi),
                 "r"(idesc), "r"(elected), "r"(acc) : "memory");
}
// arrives at the barrier when the instructions this thread has issued so far are done
__device__ __forceinline__ void umma_commit(uint32_t elected, uint32_t bar) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
               "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(bar), "r"(elected) : "memory");
}
// the 16 instructions of an item (128 codes a step, four positions each), one of its three readings
template <bool F8>
__device__ __forceinline__ void umma_item(uint32_t elected, uint32_t d, uint32_t a, uint32_t b_lo, uint32_t b_hi, uint32_t step,
                                          uint32_t half2, uint32_t idesc, uint32_t acc) {
#pragma unroll 1
  for (uint32_t end = a + 128u; a != end; a += 32u, b_lo += step) {
#pragma unroll
    for (int pp = 0; pp < 4; pp++) {
      umma<F8>(elected, d, a + pp * 8, b_lo + (uint32_t)pp * half2, b_hi, idesc, acc);
      acc = 1u;
    }
  }
}
// per-row sums T1, T2, T3 of bytes u from the three readings
struct USums { int t1, t2, t3; };
__device__ __forceinline__ USums umma_sums(uint32_t u, uint32_t s, uint32_t e) {
  USums r;
  r.t1 = ((int)u + (int)s) >> 7;
  r.t2 = ((int)u - (int)s) >> 8;
  r.t3 = (2 * r.t1 - (int)(__uint_as_float(e) * 512.f)) >> 2;   // e: (2 T1 - 4 T3) / 512, exactly
  return r;
}

__device__ __forceinline__ void sts128(uint32_t at, uint4 v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(at), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
template <int BYTES>
__device__ __forceinline__ void sts_low(uint32_t at, uint32_t v) {   // the low 1, 2 or 4 bytes of v
  if constexpr (BYTES == 4) asm volatile("st.shared.u32 [%0], %1;" ::"r"(at), "r"(v) : "memory");
  else if constexpr (BYTES == 2) asm volatile("st.shared.u16 [%0], %1;" ::"r"(at), "h"((unsigned short)v) : "memory");
  else asm volatile("st.shared.u8 [%0], %1;" ::"r"(at), "r"(v) : "memory");
}

// FQ, SDBG, LATE as in gemv_stream_kernel. PARTS: K in parts (p.part_chunks), whose activations take turns in shared memory; the
// sums stay in tensor memory, so a CTA has one tile then.
template <int FQ, bool SDBG, bool LATE, bool PARTS = false>
__global__ void __launch_bounds__(kUThreads, 1) gemv_umma_kernel(const __grid_constant__ GemvMaps maps, const UmmaParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;           // TMA 128B swizzle wants 1024-byte alignment
  uint8_t* const gen = smem_raw + (base - raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int b = blockIdx.x;
  const int M = FQ != 0 ? 1 : p.M;
  const int stages = p.stages, slots = p.slots, nbuf = p.nbuf;
  const uint32_t full0 = base + p.off_bar, empty0 = full0 + 8 * kUMaxStages, afull0 = empty0 + 8 * kUMaxStages,
                 aempty0 = afull0 + 8 * kUMaxSlots, dfull0 = aempty0 + 8 * kUMaxSlots, dempty0 = dfull0 + 8 * kUMaxBuf,
                 bfull = dempty0 + 8 * kUMaxBuf, bfree = bfull + 8, drained = bfull + 16;
  float* const s_scale = reinterpret_cast<float*>(gen + p.off_misc);    // [16], then [16] maxima of the quantizer
  int* const s_T0tot = reinterpret_cast<int*>(s_scale + 32);            // [16]: sum of q per token
  uint32_t* const s_tmem = reinterpret_cast<uint32_t*>(s_scale + 48);
  const uint32_t bs = base + (uint32_t)p.off_bs;
  const uint32_t a_col0 = 512u - 128u * (uint32_t)slots;
#ifdef RCP_CHECKED
  auto ck_fail = [&](int site) { if (p.status) atomicMax(p.status, 16 + site); };
#endif
  // The producer sets up the barriers and only announces that; the first issuer takes all of the tensor memory (which
  // therefore starts at column 0). The next kernel may start when every CTA has it, not before: one that fits beside these CTAs and
  // takes tensor memory of its own in front of its wait for this kernel would keep a CTA waiting that it waits for.
  if (warp == kUFirstIssue) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(512) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    if constexpr (!LATE) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
  // Barriers and tensor memory: the producer only announces, converters and issuers wait, the workers learn of it from the
  // first issuer when they have prepared the activations.
  auto set_up = [&]() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    asm volatile("bar.sync 3, %0;" ::"n"(kUThreads - kUWork * 32) : "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  };
  // Moves items into tensor memory, two warps to a quarter of the lanes (a warp's number modulo four says which it may write), each
  // half of an item's bytes. Where helpers join in (p.helpers), the converters (team 0) take the first items, as many as there are
  // slots, and every other one from there on.
  auto convert = [&](int team, int part) {
    int total_items = 0;
    for (int pi = 0; pi < p.nphase; pi++)
      if (b < p.phase[pi].ncta) total_items += p.phase[pi].reps * p.phase[pi].items;
    const int quad = warp & 3;
    const uint32_t row = (uint32_t)(quad * 32 + lane);
    const uint32_t a_at = a_col0 + (uint32_t)(64 * part) + ((uint32_t)(quad * 32) << 16);
    int stage = 0, slot = 0;
    uint32_t rpar = 0, apar = 1;
    bool ok = true;
    for (int it = 0; it < total_items; it++) {
      if (!p.helpers || (it < slots ? 0 : (it - slots + 1) & 1) == team) {
        ok = mbar_wait_warp(full0 + 8 * stage, rpar);
        if (!ok) break;
        const uint32_t src = base + (uint32_t)stage * kUItemBytes + row * 128u;
#pragma unroll
        for (int s = 0; s < 2; s++) {
          const uint32_t at = (uint32_t)(4 * part + 2 * s);
          const uint4 U = RCP_LDS128(src + ((at ^ (row & 7)) << 4), base, base + (uint32_t)stages * kUItemBytes, 4);
          const uint4 V = RCP_LDS128(src + (((at + 1) ^ (row & 7)) << 4), base, base + (uint32_t)stages * kUItemBytes, 4);
          const uint32_t w[8] = {U.x, U.y, U.z, U.w, V.x, V.y, V.z, V.w};
          uint32_t f[32];
#pragma unroll
          for (int i = 0; i < 8; i++) {
            f[24 + i] = w[i] & 0xC0C0C0C0u;
            f[16 + i] = (w[i] * 4u) & 0xC0C0C0C0u;
            f[8 + i] = (w[i] * 16u) & 0xC0C0C0C0u;
            f[i] = (w[i] * 64u) & 0xC0C0C0C0u;
          }
          if (s == 0) {
            ok = mbar_wait_warp(aempty0 + 8 * slot, apar);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          tmem_st32(a_at + 128u * (uint32_t)slot + 32u * s, f);
        }
        if (!ok) break;
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        // The stage is given back when what was read from it is in tensor memory, not right behind the reads: an arrival there
        // got ahead of the last of them, and where the producer was waiting for the stage (rings of two or three) that read
        // met the next item's bytes.
        if (lane == 0) {
          mbar_arrive(afull0 + 8 * slot);
          mbar_arrive(empty0 + 8 * stage);
        }
      }
      if (++slot == slots) { slot = 0; apar ^= 1u; }
      if (++stage == stages) { stage = 0; rpar ^= 1u; }
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 3);
  };

  if (warp == kUProducer) {
    // ---------------------------------------------------------------- producer (as in gemv_stream_kernel)
    if (lane == 0) {
      for (int s = 0; s < stages; s++) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, kUConv); }
      for (int s = 0; s < slots; s++) { mbar_init(afull0 + 8 * s, kUConv); mbar_init(aempty0 + 8 * s, kUIssue); }
      for (int s = 0; s < nbuf; s++) { mbar_init(dfull0 + 8 * s, kUIssue); mbar_init(dempty0 + 8 * s, (M + kUTok - 1) / kUTok * 4); }
      mbar_init(bfull, 1);
      mbar_init(bfree, kUIssue);
      mbar_init(drained, kUIssue);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncwarp();
    asm volatile("bar.arrive 3, %0;" ::"n"(kUThreads - kUWork * 32) : "memory");
    if (lane == 0) {
      int slot = 0, issued = 0;
      uint32_t par = 0;
      bool ok = true;
      const long long t_start = clock64();
      for (int pi = 0; pi < p.nphase && ok; pi++) {
        const UmmaPhase ph = p.phase[pi];
        if (b >= ph.ncta) continue;
        // of an uneven phase (one at most) the CTAs with a group less fetch no more than that: the last map is theirs
        const int fewer = ph.r > 0 && b >= ph.r ? 1 : 0;
        const CUtensorMap* const map = &maps.m[fewer ? kMaxPhases - 1 : pi];
        asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
        const uint32_t box = (uint32_t)(ph.gpc - fewer) * kGroupBytes, block = (uint32_t)ph.gpc * kGroupBytes;
        const int lo = ph.q * b + min(b, ph.r);
        for (int rp = 0; rp < ph.reps && ok; rp++) {
          const int row0 = (ph.first + rp * ph.total + lo) * 16;
          for (int it = 0; it < ph.items; it++) {
            if (issued >= stages) {
              if (!mbar_wait(empty0 + 8 * slot, par ^ 1u)) {
                if (p.status) atomicExch(p.status, 2);
                ok = false;
                break;
              }
            } else {
              const long long due = t_start + (long long)issued * p.ramp_clk;
              while (clock64() < due) { }
            }
            const uint32_t bar = full0 + 8 * slot, dst = base + (uint32_t)slot * kUItemBytes;
            const int nbox = min(ph.kp, p.nchunk - it * ph.kp);
            mbar_expect_tx(bar, (uint32_t)nbox * box);
            for (int j = 0; j < nbox; j++) {
              const int xw = (it * ph.kp + j) * kChunkWords;   // a multiple of 32 words, so 16-byte aligned
              if (RCP_CK((uint32_t)(j + 1) * block <= (uint32_t)kUItemBytes && slot < stages && (((uint32_t)j * block) & 1023u) == 0 &&
                         xw >= 0 && xw < p.K / 16 && row0 >= 0 && row0 < p.N && box > 0, 1))
                tma_load_2d(dst + (uint32_t)j * block, map, xw, row0, bar);
            }
            issued++;
            if (++slot == stages) { slot = 0; par ^= 1u; }
          }
        }
      }
      // no copy may be in flight when the CTA ends
      for (int s = 0; s < min(issued, stages); s++) mbar_wait(full0 + 8 * s, (uint32_t)((issued - s + stages - 1) / stages - 1) & 1u);
    }
    __syncwarp();
  } else if (warp >= kUFirstIssue) {
    // ---------------------------------------------------------------- issuers
    set_up();
    if (warp == kUFirstIssue) asm volatile("tcgen05.fence::before_thread_sync;\n\tbar.arrive 2, %0;" ::"n"(kUWork * 32 + 32) : "memory");
    const int which = warp - kUFirstIssue;   // 0: A unsigned, 1: A signed, 2: e4m3
    const uint32_t elected = elect_one() ? 1u : 0u;
    const uint32_t b_hi = (128u >> 4) | (1u << 14);   // eight columns further on: 128 bytes
    const uint32_t b0 = (bs >> 4) | ((uint32_t)p.bhalf << 16);
    const uint32_t step = (uint32_t)p.bstep, half2 = 2u * (uint32_t)p.bhalf, dcols = (uint32_t)p.dcols, acc_cols = (uint32_t)p.acc_cols;
    bool ok = true, ready = false;
    int slot = 0, buf = 0;
    uint32_t apar = 0, dpar = 0;
    for (int pi = 0; pi < p.nphase && ok; pi++) {
      const UmmaPhase ph = p.phase[pi];
      if (b >= ph.ncta) continue;
      const uint32_t shape = ((uint32_t)((which == 2 ? ph.ncol_f8 : ph.ncol) >> 3) << 17) | (8u << 24);   // 128 rows
      const uint32_t idesc = which == 2 ? (1u << 4) | shape                   // fp32 += e4m3 x e4m3
                                        : (2u << 4) | ((uint32_t)which << 7) | (1u << 10) | shape;   // int32 += u8 or s8 x s8
      if (!ready) { ok = mbar_wait_warp(bfull, 0); ready = true; }   // the activations, when everything else is at hand
      const int part_items = PARTS ? p.part_chunks / ph.kp : 0;   // (a multiple of kp)
      int part_left = part_items;
      uint32_t bpar = 0;
      for (int rp = 0; rp < ph.reps && ok; rp++) {
        ok = mbar_wait_warp(dempty0 + 8 * buf, dpar ^ 1u);
        const uint32_t d = (uint32_t)buf * acc_cols + (uint32_t)which * dcols;
        uint32_t b_lo = b0;
        int kp0 = 0;
        for (int it = 0; it < ph.items && ok; it++) {
          if (PARTS && part_left == 0) {   // the activations of the next part of K, in the place of these
            umma_commit(elected, bfree);
            bpar ^= 1u;
            ok = mbar_wait_warp(bfull, bpar);
            if (!ok) break;
            part_left = part_items;
            b_lo = b0;
            kp0 = 0;
          }
          ok = mbar_wait_warp(afull0 + 8 * slot, apar);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t a = a_col0 + 128u * (uint32_t)slot;
          if (which == 2) umma_item<true>(elected, d, a, b_lo, b_hi, step, half2, idesc, it > 0 ? 1u : 0u);
          else umma_item<false>(elected, d, a, b_lo, b_hi, step, half2, idesc, it > 0 ? 1u : 0u);
          umma_commit(elected, aempty0 + 8 * slot);
          if (++slot == slots) { slot = 0; apar ^= 1u; }
          if (PARTS) part_left--;
          // the next item's chunks: the next columns of this group of kpl chunks, or the next group
          kp0 += ph.kp;
          b_lo += (uint32_t)(ph.kp * (M + 1));
          if (kp0 == p.kpl) { kp0 = 0; b_lo += (uint32_t)(p.bgroup - p.kpl * (M + 1)); }
        }
        umma_commit(elected, dfull0 + 8 * buf);
        if (++buf == nbuf) { buf = 0; dpar ^= 1u; }
      }
    }
    if (!ok && lane == 0 && p.status) atomicExch(p.status, 5);
    // tensor memory is given back when nothing of this warp works on it any more
    umma_commit(elected, drained);
    __syncwarp();
    mbar_wait_warp(drained, 0);
  } else if (warp >= kUFirstConv) {
    // ---------------------------------------------------------------- converters
    set_up();
    convert(0, (warp - kUFirstConv) >> 2);
  } else {
    // ---------------------------------------------------------------- activations (workers, 512 threads)
    const int part_chunks = PARTS ? p.part_chunks : p.nchunk;
    const int R1 = M + 1;
    bool bad = false;
    if (tid < kMaxTokens) s_T0tot[tid] = 0;   // (added to behind a barrier)
    auto piece = [&](int c, int s, int pp, int h, int n) -> uint32_t {
      return bs + (uint32_t)(((c >> p.lg_kpl) * p.bgroup + s * p.bstep + (2 * pp + h) * p.bhalf + (c & (p.kpl - 1)) * R1 + n) * 16);
    };
    const bool idle = PARTS && b >= p.phase[0].ncta;   // (one phase then)
    for (int c0 = 0, part = 0; c0 < p.nchunk && !(idle && part > 0); c0 += part_chunks, part++) {   // parts of K
    const int nch = min(part_chunks, p.nchunk - c0), chunks = (nch + p.kpl - 1) >> p.lg_kpl << p.lg_kpl;   // with those that pad the last group
    if (PARTS && part > 0) {
      // the instructions on the last part's activations are done
      if (!mbar_wait_warp(bfree, (uint32_t)(part - 1) & 1u)) {
        if (lane == 0 && p.status) atomicExch(p.status, 4);
        bad = true;
      }
    }
    // the column of ones, and zeros where a chunk beyond K shares lanes with others (what the ring holds there is left over)
    for (int i = tid; i < chunks * 32; i += kUWork * 32) {
      const int c = i >> 5;
      const uint32_t v = c < nch ? 0x01010101u : 0u;
      const uint32_t at = piece(c, (i >> 3) & 3, (i >> 1) & 3, i & 1, M);
      if (RCP_CK(at >= bs && at + 16 <= bs + p.bs_bytes, 2)) sts128(at, make_uint4(v, v, v, v));
    }
    if (FQ == 0 && part == 0) asm volatile("bar.sync 1, %0;" ::"n"(kUWork * 32) : "memory");   // the totals are zero
    if constexpr (FQ != 0)
      if (tid == 0 && b * 64 < p.K) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.x + b * 64));
    if (part == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
    const int W = p.K / 16;
    if constexpr (FQ != 0) {
      unsigned* const s_amax = reinterpret_cast<unsigned*>(s_scale + 16);
      constexpr int NR = FQ > 0 ? 1 : -FQ;           // words (or parts of one) per thread
      constexpr int E = FQ > 0 ? FQ : 16;            // elements of each
      constexpr int NP = E / 2;
      float2 v[NR][NP];
      float amax;
      if constexpr (FQ > 0) amax = rotate_full_token<E>(p.x, p.inv_sqrt_b, reinterpret_cast<float*>(gen + p.off_qbuf), s_amax, v[0]);
      else amax = rotate_block_token<NR>(p.x, W, p.had_block, p.inv_sqrt_b, s_amax, v);
      const __half s16 = __float2half_rn(div_by_7(__fmul_rn(amax, p.clip_ratio)));
      const float sc = __half2float(s16);
      if (tid == 0) {
        s_scale[0] = sc;
        if (b == 0 && p.scale_out) p.scale_out[0] = s16;
      }
      const bool clamped = needs_clamp(p.clip_ratio, sc);
      int total = 0;
#pragma unroll
      for (int r = 0; r < NR; r++) {
        const int first = (r * 512 + tid) * E, w = first >> 4;   // this thread's elements: first .. first + E - 1
        if (r * 512 + warp * 32 < chunks * (kChunkWords * 16 / E)) {   // (whole warps; beyond the token: zeros)
          float2 f[NP];   // 1.5 * 2^23 + q: the low byte of the pattern is q's
          if (sc != 0.f) {
            quantize_pairs<NP>(v[r], sc, clamped, f);
          } else {
#pragma unroll
            for (int i = 0; i < NP; i++) f[i] = make_float2(12582912.f, 12582912.f);
          }
          const int c = w >> 5, s = (w >> 3) & 3, h = (w >> 2) & 1;
          uint32_t at = piece(c, s, 0, h, 0) + (uint32_t)((w & 3) * 4 + ((first >> 2) & 3));
          int tsum = 0;
          uint32_t Q[4];
#pragma unroll
          for (int pp = 0; pp < 4; pp++) {
            uint32_t d[E / 4];
#pragma unroll
            for (int j = 0; j < E / 4; j++) {
              const float2 fp = f[2 * j + (pp >> 1)];
              d[j] = __float_as_uint((pp & 1) ? fp.y : fp.x);
            }
            uint32_t q;
            if constexpr (E == 16) q = __byte_perm(__byte_perm(d[0], d[1], 0x0040), __byte_perm(d[2], d[3], 0x0040), 0x5410);
            else if constexpr (E == 8) q = __byte_perm(d[0], d[1], 0x0040) & 0xFFFFu;
            else q = d[0] & 0xFFu;
            Q[pp] = q;
            tsum = __dp4a((int)q, 0x01010101, tsum);
            const uint32_t u = (q & 0x0F0F0F0Fu) ^ 0x08080808u;
            if ((FQ > 0 || w < chunks * kChunkWords) && RCP_CK(at >= bs && at + E / 4 <= bs + p.bs_bytes, 2))
              sts_low<E / 4>(at, FQ > 0 || w < W ? u : 0u);
            at += (uint32_t)(32 * p.bhalf);
          }
          total += tsum;
          if (b == 0 && p.xq_out && w < W) {
            uint8_t* const xo = p.xq_out + (first >> 1);
            if constexpr (E == 16) *reinterpret_cast<uint2*>(xo) = make_uint2(pack_nibbles(f), pack_nibbles(f + 4));
            else if constexpr (E == 8) *reinterpret_cast<uint32_t*>(xo) = pack_nibbles(f);
            else *reinterpret_cast<uint16_t*>(xo) = (uint16_t)((Q[0] & 0xFu) | (Q[1] & 0xFu) << 4 | (Q[2] & 0xFu) << 8 | (Q[3] & 0xFu) << 12);
          }
        }
      }
      // what the quantizer's threads do not reach: zeros up to the end of the last group of chunks
      for (int i = NR * 512 * E / 64 + tid; i < chunks * 8; i += kUWork * 32) {
#pragma unroll
        for (int pp = 0; pp < 4; pp++) {
          const uint32_t at = piece(i >> 3, (i >> 1) & 3, pp, i & 1, 0);
          if (RCP_CK(at >= bs && at + 16 <= bs + p.bs_bytes, 2)) sts128(at, make_uint4(0, 0, 0, 0));
        }
      }
      total = __reduce_add_sync(0xffffffffu, total);
      if (lane == 0) atomicAdd(&s_T0tot[0], total);
    } else {
      // A unit is 64 codes of a token: 32 bytes in, a 16-byte piece for each in-byte position out. Neighbouring lanes take the
      // same codes of neighbouring tokens: their pieces are neighbours too (no bank conflicts from eight tokens on).
      const int m = lane & ((1 << p.lg_m2) - 1);
      const int units = chunks * 8, ustep = (kUWork * 32) >> p.lg_m2;
      const uint8_t* const src = p.xq + (size_t)m * (p.K / 2) + (size_t)c0 * (kChunkWords * 8);
      const int left = p.K - c0 * (kChunkWords * 16);
      int total = 0;
      constexpr int kAhead = 2;
      for (int u0 = tid >> p.lg_m2; u0 - (tid >> p.lg_m2) < units; u0 += kAhead * ustep) {   // (the same trips for the warp)
        uint4 x[kAhead][2];
#pragma unroll
        for (int i = 0; i < kAhead; i++) {
          const int u = u0 + i * ustep;
          x[i][0] = x[i][1] = make_uint4(0, 0, 0, 0);
          if (m < M && u < units && u * 64 < left) {
            x[i][0] = ld_input(reinterpret_cast<const uint4*>(src) + 2 * u);
            x[i][1] = ld_input(reinterpret_cast<const uint4*>(src) + 2 * u + 1);
          }
        }
#pragma unroll
        for (int i = 0; i < kAhead; i++) {
          const int u = u0 + i * ustep;
          if (m < M && u < units) {
            const uint32_t lo[4] = {x[i][0].x, x[i][0].z, x[i][1].x, x[i][1].z}, hi[4] = {x[i][0].y, x[i][0].w, x[i][1].y, x[i][1].w};
            const uint32_t eight = u * 64 < left ? 0x08080808u : 0u;   // (beyond K: zeros)
            uint32_t o[4][4], sum = 0;
#pragma unroll
            for (int j = 0; j < 4; j++) {
              const uint32_t p01 = __byte_perm(lo[j], hi[j], 0x6420), p23 = __byte_perm(lo[j], hi[j], 0x7531);
              o[0][j] = (p01 & 0x0F0F0F0Fu) ^ eight;
              o[1][j] = ((p01 >> 4) & 0x0F0F0F0Fu) ^ eight;
              o[2][j] = (p23 & 0x0F0F0F0Fu) ^ eight;
              o[3][j] = ((p23 >> 4) & 0x0F0F0F0Fu) ^ eight;
              sum += (o[0][j] + o[1][j]) + (o[2][j] + o[3][j]);   // bytes of at most 16 x 15
            }
            total += (int)__dp4a(sum, 0x01010101u, 0u) - (int)(eight & 15u) * 64;
            uint32_t at = piece(u >> 3, (u >> 1) & 3, 0, u & 1, m);
#pragma unroll
            for (int pp = 0; pp < 4; pp++) {
              if (RCP_CK(at >= bs && at + 16 <= bs + p.bs_bytes, 3)) sts128(at, make_uint4(o[pp][0], o[pp][1], o[pp][2], o[pp][3]));
              at += (uint32_t)(32 * p.bhalf);
            }
          }
        }
      }
#pragma unroll
      for (int d = 16; d > 0; d >>= 1)
        if (d >= (1 << p.lg_m2)) total += __shfl_xor_sync(0xffffffffu, total, d);
      if (lane < M) atomicAdd(&s_T0tot[lane], total);   // (lanes below M hold the sums of their own token: m == lane)
      if (tid < M) s_scale[tid] = __half2float(ld_input(p.scale + tid));
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the instructions read the bytes through the async proxy
    if (part == 0) {
      asm volatile("bar.sync 2, %0;" ::"n"(kUWork * 32 + 32) : "memory");
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    } else {
      asm volatile("bar.sync 1, %0;" ::"n"(kUWork * 32) : "memory");
    }
    if (tid == 0) mbar_arrive(bfull);
    }   // parts

    // ---------------------------------------------------------------- tiles' ends (workers)
    const int m0 = (warp >> 2) * kUTok;   // tokens m0 .. m0 + kUTok - 1
    if (p.helpers && warp >= 8) {
      convert(1, (warp >> 2) & 1);
    } else if (m0 < M) {
      const int quad = warp & 3, L = quad * 32 + lane, nt = min(kUTok, M - m0);
      const uint32_t t_lane = (uint32_t)(quad * 32) << 16;
      int* const red = reinterpret_cast<int*>(gen + p.off_red) + m0 * 3 * kULanes;   // [token][3][128]
      bool ok = !bad;
      int buf = 0, met = 0;   // met: tiles at whose barriers this warp has met the other three of its tokens
      uint32_t dpar = 0;
      auto finish = [&](int m, int row, uint2 lut4, const USums& t) {
        const int S3 = t.t3, S1 = t.t1 - t.t3, S2 = t.t2 - t.t3, S0 = s_T0tot[m] - S1 - S2 - S3;
        p.y[(size_t)m * p.N + row] = lut_finish(s_scale[m], lut4, S0, S1, S2, S3);
        if constexpr (SDBG) *reinterpret_cast<int4*>(p.S_out + ((size_t)m * p.N + row) * 4) = make_int4(S0, S1, S2, S3);
      };
      for (int pi = 0; pi < p.nphase && ok; pi++) {
        const UmmaPhase ph = p.phase[pi];
        if (b >= ph.ncta) continue;
        const int rows = 16 * ph.gpc;
        // this warp's lanes belong to one block of rows, or to two neighbours (16 rows a block)
        auto block_of = [&](int v) { return (v * ph.inv_rows) >> 16; };
        const int kpA = block_of(quad * 32), kpB = min(block_of(quad * 32 + 31), ph.kp - 1);
        const int kp = block_of(L);
        const bool some = kpA < ph.kp, second = kp != kpA;
        const int lo = ph.q * b + min(b, ph.r), hi = lo + ph.q + (b < ph.r ? 1 : 0);
        const int nrow0 = (hi - lo) * 16;
        for (int rp = 0; rp < ph.reps && ok; rp++) {
          const int row0 = (ph.first + rp * ph.total + lo) * 16;
          const int nrow = min(nrow0, p.N - row0);   // rows of this tile
          const int mine = ph.kp == 1 ? L : L - kp * rows;  // the row whose grid this lane fetches ahead
          const uint2 lut4 = mine < nrow ? __ldg(p.lut + row0 + mine) : make_uint2(0, 0);
          ok = mbar_wait_warp(dfull0 + 8 * buf, dpar);
#ifdef RCP_CHECKED
          // (a test's way to let this warp's wait give up)
          if (p.status && __shfl_sync(0xffffffffu, *(volatile int32_t*)p.status, 0) == -1 - warp) ok = false;
#endif
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t dA = t_lane + (uint32_t)(buf * p.acc_cols + kpA * R1), dB = dA + (uint32_t)((kpB - kpA) * R1);
          USums t[kUTok];
          if (some) {
            uint32_t o[3], o2[3], v[3][4], v2[3][4];
#pragma unroll
            for (int k = 0; k < 3; k++) {
              const uint32_t at = (uint32_t)(k * p.dcols);
              tmem_ld1(dA + at + M, o[k]);
              tmem_ld4(dA + at + m0, v[k]);
              if (kpB > kpA) {
                tmem_ld1(dB + at + M, o2[k]);
                tmem_ld4(dB + at + m0, v2[k]);
              }
            }
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (kpB > kpA && second) {
#pragma unroll
              for (int k = 0; k < 3; k++) {
                o[k] = o2[k];
#pragma unroll
                for (int i = 0; i < 4; i++) v[k][i] = v2[k][i];
              }
            }
            const USums one = umma_sums(o[0], o[1], o[2]);
#pragma unroll
            for (int i = 0; i < kUTok; i++) {
              t[i] = umma_sums(v[0][i], v[1][i], v[2][i]);
              t[i].t1 -= 8 * one.t1; t[i].t2 -= 8 * one.t2; t[i].t3 -= 8 * one.t3;
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");   // the accumulators have been read
          __syncwarp();
          if (lane == 0) mbar_arrive(dempty0 + 8 * buf);
          if (ph.kp == 1) {
#pragma unroll
            for (int i = 0; i < kUTok; i++)
              if (i < nt && L < nrow) finish(m0 + i, row0 + L, lut4, t[i]);
          } else {
            // the blocks of a row add up in shared memory
#pragma unroll
            for (int i = 0; i < kUTok; i++)
              if (i < nt && kp < ph.kp && RCP_CK(((m0 + i) * 3 + 3) * kULanes * 4 <= p.red_bytes, 12)) {
                red[(i * 3 + 0) * kULanes + L] = t[i].t1;
                red[(i * 3 + 1) * kULanes + L] = t[i].t2;
                red[(i * 3 + 2) * kULanes + L] = t[i].t3;
              }
            asm volatile("bar.sync %0, 128;" ::"r"(4 + (warp >> 2)) : "memory");
            for (int e = L; e < rows * nt; e += kULanes) {
              const int i = block_of(e), rr = e - i * rows;
              if (rr < nrow) {
                USums a = {0, 0, 0};
                const int* d = red + i * 3 * kULanes + rr;
#pragma unroll 4
                for (int k = 0; k < ph.kp; k++, d += rows) { a.t1 += d[0]; a.t2 += d[kULanes]; a.t3 += d[2 * kULanes]; }
                finish(m0 + i, row0 + rr, rr == mine ? lut4 : __ldg(p.lut + row0 + rr), a);
              }
            }
            asm volatile("bar.sync %0, 128;" ::"r"(4 + (warp >> 2)) : "memory");
            met++;
          }
          if (++buf == nbuf) { buf = 0; dpar ^= 1u; }
        }
      }
      if (!ok) {
        if (lane == 0 && p.status) atomicExch(p.status, 3);
        // the other three may have made it: they are not left alone at the barriers of the tiles still to come
        int left = -2 * met;   // (two a tile)
#pragma unroll 1
        for (int pi = 0; pi < p.nphase; pi++)
          if (b < p.phase[pi].ncta && p.phase[pi].kp > 1) left += 2 * p.phase[pi].reps;
#pragma unroll 1
        for (; left > 0; left--) asm volatile("bar.sync %0, 128;" ::"r"(4 + (warp >> 2)) : "memory");
      }
    }
  }
  // When the next kernel may start: as in gemv_stream_kernel.
  if constexpr (LATE) asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kUFirstIssue) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(0), "r"(512) : "memory");
  }
}

}  // namespace rcp
