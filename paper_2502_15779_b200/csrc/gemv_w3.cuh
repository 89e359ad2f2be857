// 3-bit weights (Section 4.3, paragraph "Application of LDP on NF3 format"; Table "memory", W3 column):
// packing and the W3A4 look-up-table GEMV with eight levels per quantization unit.
//
// Storage. The low two bits of a code are stored exactly like a 2-bit code (words2 [N][K/16]); the top bit goes
// to a plane of its own (words1 [N][K/32]): word v covers the codes 32v .. 32v+31 and holds the top bit of code
// 32v + i in bit 2i and of code 32v + 16 + i in bit 2i + 1. Masked with 0x55555555 (shifted down by one for the
// second half) a plane word therefore lines up with the b0 bits of the matching words2 word.
//
// Exact integer formulation. With b0, b1, b2 the bits of a code, the sums of q over the seven products
//   b0, b1, b0 b1, b2, b0 b2, b1 b2, b0 b1 b2      (T_S for the non-empty subsets S of {0,1,2})
// and T_0 = sum of q give every per-code sum by inclusion and exclusion:
//   S_c = sum over S containing the set bits of c of (-1)^(|S| - popcount(c)) T_S.
// Each product is a bit plane of 16 single bits (one logic operation per plane and word); masked at in-byte
// position p it is the A operand of an 8-bit dot product (dp4a) against the int8 activations, even positions
// meeting activations pre-multiplied by 4 so that positions {0,1} and {2,3} share an accumulator.
// 2.4 times the mask and dot-product work of the 2-bit kernel per weight. One warp per output row, lanes along
// K in units of 64 codes (a 16-byte and an 8-byte load), two units = one group of 128 per lane step; one resident
// wave of CTAs, rows dealt round-robin to its warps.
#pragma once
#include "common.cuh"

namespace rcp {

__global__ void pack_weights3_kernel(const uint4* __restrict__ codes, size_t nplane, uint32_t* __restrict__ words2,
                                     uint32_t* __restrict__ words1, int* __restrict__ bad) {
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < nplane; v += (size_t)gridDim.x * blockDim.x) {
    const uint4 a = __ldg(codes + 2 * v), b = __ldg(codes + 2 * v + 1);   // codes 32v .. 32v+15, 32v+16 .. 32v+31
    const uint32_t c[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint32_t lo[2] = {0, 0}, top = 0, over = 0;
#pragma unroll
    for (int i = 0; i < 8; i++) {
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const uint32_t code = (c[i] >> (8 * j)) & 0xFFu;
        const int k = 4 * i + j;                       // 0..31 inside the plane word
        over |= code & ~7u;
        lo[k >> 4] |= (code & 3u) << (2 * (k & 15));
        top |= ((code >> 2) & 1u) << (k < 16 ? 2 * k : 2 * (k - 16) + 1);
      }
    }
    words2[2 * v] = lo[0];
    words2[2 * v + 1] = lo[1];
    words1[v] = top;
    if (over) atomicExch(bad, 1);
  }
}

// Export of a 3-bit layer trained with a learnable centre (Section 4.3, paragraph "Application of LDP on NF3
// format", Eq. "nf3scales", Eq. "nf3") to the inputs of the kernel below: packed codes and the eight levels of
// every quantization unit. Offline, one pass: 2 bytes read and 3/8 byte written per weight. One warp per unit
// (G consecutive weights of a row, G a multiple of 32): the range by shuffles; centre, the two scales and the
// levels in fp32 with one rounding per operation, so that the 3-bit decision is reproducible bit for bit; a
// lane takes four consecutive weights per round of 128, four lanes make a word of low bits, eight lanes a word
// of the top-bit plane. `table`: the eight ascending normalized levels of the format, table[zero] == 0.
struct Nf3Params {
  const __half* w;     // [N][K] rotated weights
  const float* sb;     // [N][K/G] sigmoid(beta): lower clipping fraction
  const float* sg;     // sigmoid(gamma)
  const float* s1;     // sigmoid(s_1): the centre as a fraction of the clipped range
  uint32_t* words2;    // [N][K/16]
  uint32_t* words1;    // [N][K/32]
  uint4* lut;          // [N][K/G] eight fp16 levels
  float table[8];
  int zero;
  int N, K, G;
  long long units;     // N * K / G
};

__global__ void __launch_bounds__(256) nf3_export_kernel(const Nf3Params p) {
  const int lane = threadIdx.x & 31;
  const long long warp0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const int NG = p.K / p.G;
  for (long long u = warp0; u < p.units; u += nwarps) {
    const long long n = u / NG;
    const int j = (int)(u - n * NG);
    const __half* wu = p.w + n * p.K + (long long)j * p.G;
    float wmin = INFINITY, wmax = -INFINITY;
    for (int k0 = lane * 4; k0 < p.G; k0 += 128) {
      const uint2 raw = __ldg(reinterpret_cast<const uint2*>(wu + k0));
      const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
      const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
      wmin = fminf(fminf(wmin, fminf(a.x, a.y)), fminf(b.x, b.y));
      wmax = fmaxf(fmaxf(wmax, fmaxf(a.x, a.y)), fmaxf(b.x, b.y));
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
      wmin = fminf(wmin, __shfl_xor_sync(0xffffffffu, wmin, d));
      wmax = fmaxf(wmax, __shfl_xor_sync(0xffffffffu, wmax, d));
    }
    const float lo = __fmul_rn(__ldg(p.sb + u), wmin);
    const float hi = __fmul_rn(__ldg(p.sg + u), wmax);
    const float h = __fsub_rn(hi, lo);
    const float c = __fadd_rn(lo, __fmul_rn(h, __ldg(p.s1 + u)));
    const float s_neg = fabsf(__fsub_rn(c, lo)), s_pos = fabsf(__fsub_rn(hi, c));
    const bool ok = h > 0.0f;
    if (lane < 8) {   // lane i makes level i; the eight halves are gathered into one 16-byte store
      const float level = __fadd_rn(c, __fmul_rn(p.table[lane], lane > p.zero ? s_pos : s_neg));
      const uint32_t bits = __half_as_ushort(__float2half_rn(ok ? level : lo));
      const uint32_t other = __shfl_down_sync(0x000000ffu, bits, 1, 8);
      const uint32_t pair = bits | (other << 16);                    // valid in even lanes
      uint4 out;
      out.x = __shfl_sync(0x000000ffu, pair, 0);
      out.y = __shfl_sync(0x000000ffu, pair, 2);
      out.z = __shfl_sync(0x000000ffu, pair, 4);
      out.w = __shfl_sync(0x000000ffu, pair, 6);
      if (lane == 0) p.lut[u] = out;
    }
    __syncwarp();
    uint32_t* row2 = p.words2 + n * (p.K / 16) + (long long)j * (p.G / 16);
    uint32_t* row1 = p.words1 + n * (p.K / 32) + (long long)j * (p.G / 32);
    for (int k0 = lane * 4; k0 - lane * 4 < p.G; k0 += 128) {   // all lanes stay in the loop for the shuffles
      uint32_t low = 0, top = 0;
      if (k0 < p.G) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2*>(wu + k0));
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
        const float v[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
        for (int e = 0; e < 4; e++) {
          int code = p.zero;
          if (ok) {
            const float cl = fminf(fmaxf(v[e], lo), hi);
            const bool pos = cl > c;            // a weight equal to the centre belongs to the negative side
            const float sc = pos ? s_pos : s_neg;
            if (sc > 0.0f) {
              const float x = __fdiv_rn(__fsub_rn(cl, c), sc);
              const int first = pos ? p.zero : 0, last = pos ? 7 : p.zero;
              code = first;
              float best = fabsf(__fsub_rn(x, p.table[first]));
              for (int i = first + 1; i <= last; i++) {
                const float dist = fabsf(__fsub_rn(x, p.table[i]));
                if (dist < best) { best = dist; code = i; }   // strict: a tie keeps the lower level
              }
            }
          }
          low |= (uint32_t)(code & 3) << (2 * e);
          const int kk = (k0 + e) & 31;       // place in the plane word: codes 0..15 even bits, 16..31 odd bits
          top |= (uint32_t)(code >> 2) << (kk < 16 ? 2 * kk : 2 * (kk - 16) + 1);
        }
      }
      uint32_t word = low << (8 * (lane & 3));
      word |= __shfl_xor_sync(0xffffffffu, word, 1);
      word |= __shfl_xor_sync(0xffffffffu, word, 2);
      top |= __shfl_xor_sync(0xffffffffu, top, 1);
      top |= __shfl_xor_sync(0xffffffffu, top, 2);
      top |= __shfl_xor_sync(0xffffffffu, top, 4);
      if ((lane & 3) == 0 && k0 < p.G) row2[k0 >> 4] = word;
      if ((lane & 7) == 0 && k0 < p.G) row1[k0 >> 5] = top;
    }
  }
}

constexpr int kW3Threads = 256;

struct W3Params {
  const uint32_t* words2;
  const uint32_t* words1;
  const uint4* lut;        // [N][8] fp16 (GRP: [N][K/128][8])
  const uint8_t* xq;       // [K/2] of the token
  const __half* scale;     // of the token
  __half* y;               // [N] of the token
  int32_t* S_out;          // SDBG: [N][8] (GRP: [N][K/128][8]) of the token
  int N, K;
};

// S_c from the eight subset sums (index = bit set of the subset; t[0] = sum of q)
__device__ __forceinline__ void w3_percode(const int (&t)[8], int (&S)[8]) {
  S[7] = t[7];
  S[6] = t[6] - t[7];
  S[5] = t[5] - t[7];
  S[3] = t[3] - t[7];
  S[4] = t[4] - t[5] - t[6] + t[7];
  S[2] = t[2] - t[3] - t[6] + t[7];
  S[1] = t[1] - t[3] - t[5] + t[7];
  S[0] = t[0] - t[1] - t[2] - t[4] + t[3] + t[5] + t[6] - t[7];
}

__device__ __forceinline__ float w3_lut_dot(uint4 l, const int (&S)[8]) {
  const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&l.x));
  const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&l.y));
  const float2 c = __half22float2(*reinterpret_cast<const __half2*>(&l.z));
  const float2 d = __half22float2(*reinterpret_cast<const __half2*>(&l.w));
  float acc = a.x * (float)S[0];
  acc = fmaf(a.y, (float)S[1], acc);
  acc = fmaf(b.x, (float)S[2], acc);
  acc = fmaf(b.y, (float)S[3], acc);
  acc = fmaf(c.x, (float)S[4], acc);
  acc = fmaf(c.y, (float)S[5], acc);
  acc = fmaf(d.x, (float)S[6], acc);
  acc = fmaf(d.y, (float)S[7], acc);
  return acc;
}

// Four 4-bit two's-complement values, one in the low nibble of each byte (high nibbles zero), sign-extended to
// bytes: with t = v ^ 8 per byte the result is t - 8; the bytes are lifted to 0x80 + t first so that no borrow
// crosses a byte, and the lift is taken out again.
__device__ __forceinline__ uint32_t w3_sext4x4(uint32_t v) {
  return (((v ^ 0x08080808u) | 0x80808080u) - 0x08080808u) ^ 0x80808080u;
}
// a & b & MASK as one logic operation with the mask as an immediate
template <uint32_t MASK>
__device__ __forceinline__ uint32_t w3_and_mask(uint32_t a, uint32_t b) {
  uint32_t d;
  asm("lop3.b32 %0, %1, %2, %3, 0x80;" : "=r"(d) : "r"(a), "r"(b), "n"(MASK));
  return d;
}
// In-byte position PP of a word: the seven products of code bits and their dot products. w: the word (b0 in the even, b1 in
// the odd bits), s = 2 w (b0 in the odd bits), ws = w & s (b0 b1 there), Z: b2 in the odd bits. All but b0 are taken at the
// odd bit of the position, where a plane word's second half stands as it is and its first half after one addition, so no
// right shift is needed (additions run on either of two pipes, shifts and logic on one, which bounds this kernel); the
// other bits drop out under the mask. Position 3 sits in bits 6 and 7: one mask keeps both, and read as unsigned and as
// signed bytes it weighs 64 b0 + 128 b1 and 64 b0 - 128 b1, which gives b0 and b1 (accP).
template <int PP>
__device__ __forceinline__ void w3_position(uint32_t w, uint32_t s, uint32_t ws, uint32_t Z, uint32_t q, int (&acc)[7][2],
                                            int (&accP)[2]) {
  constexpr uint32_t m0 = 0x01010101u << (2 * PP), m1 = m0 << 1;
  if constexpr (PP < 3) {
    dp4a_u8s8(acc[0][PP >> 1], w & m0, q);                        // b0
    dp4a_u8s8(acc[1][PP >> 1], w & m1, q);                        // b1, times 2 like all that follow
  } else {
    const uint32_t both = w & 0xC0C0C0C0u;
    dp4a_u8s8(accP[0], both, q);
    dp4a_s8s8(accP[1], both, q);
  }
  dp4a_u8s8(acc[2][PP >> 1], ws & m1, q);                         // b0 b1
  dp4a_u8s8(acc[3][PP >> 1], Z & m1, q);                          // b2
  dp4a_u8s8(acc[4][PP >> 1], w3_and_mask<m1>(s, Z), q);           // b0 b2
  dp4a_u8s8(acc[5][PP >> 1], w3_and_mask<m1>(w, Z), q);           // b1 b2
  dp4a_u8s8(acc[6][PP >> 1], w3_and_mask<m1>(ws, Z), q);          // b0 b1 b2
}
// the subset sums t[0..6] (b0, b1, b0 b1, b2, b0 b2, b1 b2, b0 b1 b2) from the accumulators
__device__ __forceinline__ void w3_subset_sums(const int (&acc)[7][2], const int (&accP)[2], int (&t)[7]) {
  t[0] = (acc[0][0] >> 2) + (acc[0][1] >> 6) + ((accP[0] + accP[1]) >> 7);
  t[1] = (acc[1][0] >> 3) + (acc[1][1] >> 7) + ((accP[0] - accP[1]) >> 8);
#pragma unroll
  for (int f = 2; f < 7; f++) t[f] = (acc[f][0] >> 3) + (acc[f][1] >> 7);
}

// One token per launch. Shared memory: the token's activations expanded to one byte per code, 16 bytes per
// word of 16 codes: { position 0 (times 4), position 1, position 2 (times 4), position 3 }, byte j of a position =
// activation of code 16 w + 4 j + p. A lane step covers 64 units of 64 codes; lane l takes units 2l and 2l + 1 of it (128
// consecutive codes, one group of the group-wise grid; HALF: units l and l + 32), i.e. eight words c = 0..7. Word c of lane l in
// step `it` sits at 16-byte slot (it * 8 + c) * 32 + l: the lanes of a warp read consecutive slots (no bank
// conflicts) at offsets from one address that are known at compile time. K is padded to whole lane steps with
// zeros (weights beyond K are loaded as zeros as well, so the padding contributes nothing).
// Four CTAs per SM (64 registers, no spills): 32 warps hide the weight loads better than the 24 that the
// compiler's own choice of 80 registers leaves (57344x8192: 74.5 against 76.8 us).
//   HALF: where the last step of a row is at most half full (K = 14336 is three and a half steps), every lane has a unit of
// each half, and the empty half is left out by the whole warp: 4096x14336 15.1 -> 13.9 us. A form of its own, because the
// branch costs spills at 64 registers (57344x8192 would take 74.7 us instead of 69.1).
//   A warp's (row, lane step) pairs are one sequence, worked on from two buffers in turn, the weights of the next pair on
// their way. A finished row leaves its seven sums in shared memory; the eight-level dot products are done for up to 32 rows
// at once, one per lane. (One lane finishing one row at a time was a tenth of the instructions at K = 4096 and, with them,
// its latency once a row: 28672x4096 23.1 -> 20.9 us, 57344x8192 74.2 -> 70.6.)
template <bool GRP, bool SDBG, bool HALF>
__global__ void __launch_bounds__(kW3Threads, 4) gemv_w3a4_kernel(const W3Params p) {
  extern __shared__ uint4 s_act[];           // [lane steps][8][32]
  constexpr int kWarps = kW3Threads / 32;
  __shared__ int s_t0[kWarps];
  __shared__ int s_t0g[GRP ? 512 : 1];       // sum of q per group of 128 (K <= 65536)
  __shared__ int4 s_sum[GRP ? 1 : kWarps][GRP ? 1 : 32][2];   // sums of the rows that wait to be finished
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int W = p.K / 16;
  const int nunit = p.K / 64;
  const int nit = (nunit + 63) / 64;         // lane steps per row
  const int warps = gridDim.x * kWarps;
  static_assert(!(GRP && HALF), "the group-wise grid wants both units of a group in one lane");
  const int unit0 = HALF ? lane : 2 * lane;   // a lane's units in a step: unit0 and unit0 + unit_h
  constexpr int unit_h = HALF ? 32 : 1;
  struct Step { uint4 a[2]; uint2 z[2]; };   // the weights of a lane step: two units, each one uint4 of words2, one uint2 of words1
  auto fetch = [&](int row, int it, Step& d) {
    const int u = unit0 + 64 * it;
    const size_t e = (size_t)row * nunit + u;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const bool ok = row < p.N && u + h * unit_h < nunit;
      d.a[h] = ok ? ld_input(reinterpret_cast<const uint4*>(p.words2) + e + h * unit_h) : make_uint4(0, 0, 0, 0);
      d.z[h] = ok ? ld_input(reinterpret_cast<const uint2*>(p.words1) + e + h * unit_h) : make_uint2(0, 0);
    }
  };
  // Rows are dealt round-robin to all warps of the grid (one resident wave of CTAs). Launched with programmatic stream
  // serialization: nothing is read before the wait (the kernel in front may be the export of this very layer), but the
  // first weights are sent on their way to L2, which is where such a kernel would put them (4096x14336: 15.7 -> 15.4 us).
  const int gw = blockIdx.x * kWarps + warp;
  Step A, B;
  if (gw < p.N && unit0 < nunit) {
    const size_t e = (size_t)gw * nunit + unit0;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p.words2 + 4 * e));
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p.words1 + 2 * e));
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  fetch(gw, 0, A);
  // ---- expand the activations (256 words per lane step: the same trip count for every thread)
  int tsum = 0;
  for (int w = tid; w < nit * 256; w += kW3Threads) {
    uint2 x = make_uint2(0, 0);
    if (w < W) x = ld_input(reinterpret_cast<const uint2*>(p.xq) + w);   // 16 nibbles
    // four nibbles at a time: nibble k of a register goes to byte k / 2 of e (k even) or o (k odd), is sign-extended
    // inside its byte, then the bytes are gathered by position (byte j of position pp = code 4 j + pp)
    const uint32_t e0 = w3_sext4x4(x.x & 0x0F0F0F0Fu), o0 = w3_sext4x4((x.x >> 4) & 0x0F0F0F0Fu);   // codes 0,2,4,6 / 1,3,5,7
    const uint32_t e1 = w3_sext4x4(x.y & 0x0F0F0F0Fu), o1 = w3_sext4x4((x.y >> 4) & 0x0F0F0F0Fu);   // codes 8,.. / 9,..
    uint4 pos;
    pos.x = (__byte_perm(e0, e1, 0x6420) << 2) & 0xFCFCFCFCu;   // codes 0,4,8,12, times 4 inside each byte
    pos.y = __byte_perm(o0, o1, 0x6420);                        // codes 1,5,9,13
    pos.z = (__byte_perm(e0, e1, 0x7531) << 2) & 0xFCFCFCFCu;   // codes 2,6,10,14, times 4
    pos.w = __byte_perm(o0, o1, 0x7531);                        // codes 3,7,11,15
    int wsum = __dp4a((int)e0, 0x01010101, __dp4a((int)o0, 0x01010101, __dp4a((int)e1, 0x01010101, __dp4a((int)o1, 0x01010101, 0))));
    // word c = 4 h + i of lane l in step w >> 8: word i of its unit h
    if constexpr (HALF) s_act[((w >> 7) * 4 + (w & 3)) * 32 + ((w >> 2) & 31)] = pos;
    else s_act[((w >> 8) * 8 + (w & 7)) * 32 + ((w >> 3) & 31)] = pos;
    if constexpr (GRP) {
      // eight consecutive words are one group; they belong to eight consecutive lanes
      wsum += __shfl_xor_sync(0xffffffffu, wsum, 1);
      wsum += __shfl_xor_sync(0xffffffffu, wsum, 2);
      wsum += __shfl_xor_sync(0xffffffffu, wsum, 4);
      if (w < W && (w & 7) == 0) s_t0g[w >> 3] = wsum;
    } else {
      tsum += wsum;
    }
  }
  if constexpr (!GRP) {
    tsum = __reduce_add_sync(0xffffffffu, tsum);
    if (lane == 0) s_t0[warp] = tsum;
  }
  __syncthreads();
  int T0 = 0;
  if constexpr (!GRP) {
#pragma unroll
    for (int i = 0; i < kWarps; i++) T0 += s_t0[i];
  }
  const float s = __half2float(p.scale[0]);
  const int ngrp = p.K / 128;
  // The arithmetic of a lane step into the fourteen accumulators (weights beyond K are zeros: no guard needed).
  int acc[7][2], accP[2];
  auto clear = [&]() {
#pragma unroll
    for (int f = 0; f < 7; f++) { acc[f][0] = 0; acc[f][1] = 0; }
    accP[0] = 0;
    accP[1] = 0;
  };
  clear();
  const uint4* const act_lane = s_act + lane;
  auto lane_step = [&](const Step& c, int it) {
    const uint4* const act = act_lane + it * 256;
#pragma unroll
    for (int h = 0; h < 2; h++) {
      if (HALF && h == 1 && 64 * it + 32 >= nunit) break;
      const uint32_t ww[4] = {c.a[h].x, c.a[h].y, c.a[h].z, c.a[h].w};
#pragma unroll
      for (int i = 0; i < 4; i++) {
        const uint32_t w = ww[i], s = w + w, ws = w & s;
        const uint32_t z = (i < 2) ? c.z[h].x : c.z[h].y;
        const uint32_t Z = (i & 1) ? z : z + z;   // the plane word's first half is in its even bits, the second in the odd ones
        const uint4 q = act[(h * 4 + i) * 32];
        w3_position<0>(w, s, ws, Z, q.x, acc, accP);
        w3_position<1>(w, s, ws, Z, q.y, acc, accP);
        w3_position<2>(w, s, ws, Z, q.z, acc, accP);
        w3_position<3>(w, s, ws, Z, q.w, acc, accP);
      }
    }
  };
  // Group-wise grid: this lane's 128 codes of step `it` are group lane + 32 it of the row; its term of y.
  auto finish_group = [&](int row, int it) -> float {
    const int gi = lane + 32 * it;
    int sums[7], t[8], S[8];
    w3_subset_sums(acc, accP, sums);
    clear();
#pragma unroll
    for (int f = 0; f < 7; f++) t[f + 1] = sums[f];
    if (gi >= ngrp) return 0.f;
    t[0] = s_t0g[GRP ? gi : 0];
    w3_percode(t, S);
    if constexpr (SDBG) {
      int4* o = reinterpret_cast<int4*>(p.S_out + ((size_t)row * ngrp + gi) * 8);
      o[0] = make_int4(S[0], S[1], S[2], S[3]);
      o[1] = make_int4(S[4], S[5], S[6], S[7]);
    }
    return w3_lut_dot(ld_input(p.lut + (size_t)row * ngrp + gi), S);
  };
  // Per-row grid: the rows first, first + warps, .. (cnt of them), one per lane, from their sums.
  auto finish_rows = [&](int first, int cnt) {
    __syncwarp();
    if (lane < cnt) {
      const int row = first + lane * warps;
      const int4 lo = s_sum[warp][lane][0], hi = s_sum[warp][lane][1];
      const int t[8] = {T0, lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z};
      int S[8];
      w3_percode(t, S);
      p.y[row] = __float2half_rn(s * w3_lut_dot(ld_input(p.lut + row), S));
      if constexpr (SDBG) {
        int4* o = reinterpret_cast<int4*>(p.S_out + (size_t)row * 8);
        o[0] = make_int4(S[0], S[1], S[2], S[3]);
        o[1] = make_int4(S[4], S[5], S[6], S[7]);
      }
    }
    __syncwarp();
  };
  float yacc = 0.f;
  int row = gw, it = 0, first = gw, cnt = 0;
  // One pair: asks for the next one's weights, works on this one's; false after the warp's last.
  auto step = [&](const Step& c, Step& next) -> bool {
    const bool last = it + 1 == nit;
    const int nrow = last ? row + warps : row, nxt = last ? 0 : it + 1;
    fetch(nrow, nxt, next);
    lane_step(c, it);
    if constexpr (GRP) {
      yacc += finish_group(row, it);
      if (last) {
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) yacc += __shfl_xor_sync(0xffffffffu, yacc, d);
        if (lane == 0) p.y[row] = __float2half_rn(s * yacc);
        yacc = 0.f;
      }
    } else if (last) {
      int t[7];
      w3_subset_sums(acc, accP, t);
      clear();
#pragma unroll
      for (int f = 0; f < 7; f++) t[f] = __reduce_add_sync(0xffffffffu, t[f]);   // one instruction per sum
      if (lane == 0) {
        s_sum[warp][cnt][0] = make_int4(t[0], t[1], t[2], t[3]);
        s_sum[warp][cnt][1] = make_int4(t[4], t[5], t[6], 0);
      }
      if (++cnt == 32) {
        finish_rows(first, cnt);
        first = nrow;
        cnt = 0;
      }
    }
    row = nrow;
    it = nxt;
    return row < p.N;
  };
  if (row < p.N)
    while (step(A, B) && step(B, A)) { }
  // Only now: CTAs of the next kernel that come to wait beside busy ones cost them more than their early start returns
  // (1000x1024 in a chain 4.1 us with the trigger at the start, 2.4 here, 2.8 with a plain launch).
  asm volatile("griddepcontrol.launch_dependents;");
  if constexpr (!GRP) finish_rows(first, cnt);
}

}  // namespace rcp
