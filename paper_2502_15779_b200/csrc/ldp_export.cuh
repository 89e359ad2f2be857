// Export of a layer trained with learnable direct partitioning to the GEMV's inputs (Section 4.3:
// Eq. "partition", the grid t_i, Eq. "quant", Eq. "dequantgrid"; Section 4.4 Eq. "deqgrid"; the
// clipping range of Section 4.2). An offline, one-pass kernel: 2 bytes read and a quarter byte
// written per weight. One warp per quantization unit (G consecutive weights of a row): the range by
// shuffles, the three thresholds and four levels in fp32 with one rounding per operation (so the
// 2-bit decision is reproducible bit for bit), codes packed 16 to a word straight away.
#pragma once
#include <type_traits>

#include "common.cuh"

namespace rcp {

struct LdpParams {
  const __half* w;     // [N][K] rotated weights
  const float* sb;     // [N][K/G] sigmoid(beta): lower clipping fraction
  const float* sg;     // sigmoid(gamma)
  const float* s1;     // sigmoid(s_1)
  const float* s2;     // sigmoid(s_2)
  uint32_t* words;     // [N][K/16]
  uint2* lut;          // [N][K/G] four fp16 levels
  int N, K, G;
  long long units;     // N * K / G
};

__global__ void __launch_bounds__(256) ldp_export_kernel(const LdpParams p) {
  const int lane = threadIdx.x & 31;
  const long long warp0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const int NG = p.K / p.G;
  for (long long u = warp0; u < p.units; u += nwarps) {
    const long long n = u / NG;
    const int j = (int)(u - n * NG);
    const __half* wu = p.w + n * p.K + (long long)j * p.G;
    // range of the unit: a lane takes 4 consecutive weights per round of 128
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
    const float p1 = __ldg(p.s1 + u), r2 = __ldg(p.s2 + u);
    const float rest = __fsub_rn(1.0f, p1);
    const float p2 = __fmul_rn(rest, r2);
    const float p3 = __fmul_rn(rest, __fsub_rn(1.0f, r2));
    const float t1 = __fdiv_rn(p1, 2.0f);
    const float t2 = __fadd_rn(t1, __fdiv_rn(__fadd_rn(p1, p2), 2.0f));
    const float t3 = __fadd_rn(t2, __fdiv_rn(__fadd_rn(p2, p3), 2.0f));
    const bool ok = h > 0.0f;
    if (lane == 0) {
      const float w1 = __fdiv_rn(__fadd_rn(t1, t2), 2.0f), w2 = __fdiv_rn(__fadd_rn(t2, t3), 2.0f);
      float lv[4] = {__fadd_rn(lo, __fmul_rn(h, 0.0f)), __fadd_rn(lo, __fmul_rn(h, w1)), __fadd_rn(lo, __fmul_rn(h, w2)), __fadd_rn(lo, __fmul_rn(h, 1.0f))};
      if (!ok) lv[0] = lv[1] = lv[2] = lv[3] = lo;
      const __half2 l01 = __halves2half2(__float2half_rn(lv[0]), __float2half_rn(lv[1]));
      const __half2 l23 = __halves2half2(__float2half_rn(lv[2]), __float2half_rn(lv[3]));
      uint2 out;
      out.x = *reinterpret_cast<const uint32_t*>(&l01);
      out.y = *reinterpret_cast<const uint32_t*>(&l23);
      p.lut[u] = out;
    }
    // codes: 4 per lane, 16 per group of four lanes = one packed word
    uint32_t* wordrow = p.words + n * (p.K / 16) + (long long)j * (p.G / 16);
    for (int k0 = lane * 4; k0 - lane * 4 < p.G; k0 += 128) {   // all lanes stay in the loop for the shuffles
      uint32_t byte = 0;
      if (k0 < p.G && ok) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2*>(wu + k0));
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
        const float v[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
        for (int e = 0; e < 4; e++) {
          const float c = fminf(fmaxf(v[e], lo), hi);
          const float x = __fdiv_rn(__fsub_rn(c, lo), h);
          const uint32_t code = (uint32_t)(x >= t1) + (uint32_t)(x >= t2) + (uint32_t)(x >= t3);
          byte |= code << (2 * e);
        }
      }
      uint32_t word = byte << (8 * (lane & 3));
      word |= __shfl_xor_sync(0xffffffffu, word, 1);
      word |= __shfl_xor_sync(0xffffffffu, word, 2);
      if ((lane & 3) == 0 && k0 < p.G) wordrow[k0 >> 4] = word;
    }
  }
}

// ---------------------------------------------------------------------------------------------
// The same export for units of 128 weights (the paper's group size), where it has to move 2.4 bytes per weight and
// the kernel above spends its time on arithmetic instead: an IEEE division, two clampings and three comparisons
// per weight, and ten shuffles for every four weights of a lane.
//   The code of a weight is a non-decreasing function of the weight (clamping, subtraction and division by
// h > 0 all are, their roundings included), and the weight is an fp16 number. So every threshold t_i has a smallest
// fp16 value c_i whose quotient reaches it, and code = number of c_i <= w exactly, whatever the roundings: three
// packed half comparisons per two weights, no division. c_i comes from lo + t_i h and is then checked against the
// definition itself (c_i reaches t_i, its predecessor does not); where that first guess is off by more than one
// value, a bisection over the fp16 numbers finds it.
//   A warp takes 32 units = 4096 consecutive weights (units are consecutive in memory whatever K is) and keeps them
// in registers, 16 vectors of 8 weights per lane, so they are read once, the next tile being copied to shared memory
// meanwhile. Per-unit minima and maxima meet in a transposing reduction (15 exchanges for 16 values instead of 4 per
// value), which leaves lane l with unit
// 2 (l & 15) + (l >> 4): the per-unit arithmetic runs once per unit, one unit per lane. About 8 instructions per
// weight against 40. 28672 x 4096 weights: 52.7 us, 415 with the kernel above (memory floor 44).
constexpr int kLdpGroup = 128;

// value number k of the fp16 numbers in ascending order (k = 0: zero; k = +-0x7C00: the infinities)
__device__ __forceinline__ __half half_of_key(int k) {
  return __ushort_as_half((unsigned short)(k >= 0 ? k : 0x8000 - k));
}
__device__ __forceinline__ int key_of_half(__half h) {
  const int b = __half_as_ushort(h);
  return b & 0x8000 ? -(b & 0x7FFF) : b;
}
// whether the fp16 number with key k, clamped to [lo, hi], has reached threshold t (the definition, rounding by rounding)
__device__ __forceinline__ bool ldp_reached(int k, float lo, float hi, float h, float t) {
  const float c = fminf(fmaxf(__half2float(half_of_key(k)), lo), hi);
  return __fdiv_rn(__fsub_rn(c, lo), h) >= t;
}
// key of the smallest fp16 number that has reached t; 0x7C01 (a NaN, which no weight reaches) where none has
__device__ __forceinline__ int ldp_cut(float lo, float hi, float h, float t) {
  const int k = key_of_half(__float2half_rn(fminf(fmaxf(fmaf(t, h, lo), lo), hi)));
  const bool at = ldp_reached(k, lo, hi, h, t);
  if (at && !ldp_reached(k - 1, lo, hi, h, t)) return k;
  if (!at && ldp_reached(k + 1, lo, hi, h, t)) return k + 1;
  int a = -0x7C01, b = 0x7C01;   // the guess is not within one value: bisect (up to a: not reached; from b on: reached)
  while (b - a > 1) {
    const int m = (a + b) >> 1;
    if (ldp_reached(m, lo, hi, h, t)) b = m; else a = m;
  }
  return b;
}

constexpr int kLdpWarps = 8;
constexpr size_t kLdpSmem = (size_t)kLdpWarps * 32 * kLdpGroup * 2;   // a tile of 32 units per warp

__global__ void __launch_bounds__(kLdpWarps * 32, 2) ldp_export128_kernel(const LdpParams p) {
  extern __shared__ __align__(16) uint4 s_tile[];   // [warp][step][lane]: every lane reads what it copied itself
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long ntile = (p.units + 31) / 32, stride = (long long)gridDim.x * kLdpWarps;
  uint4* const mybuf = s_tile + warp * 512 + lane;
  const int mine = 2 * (lane & 15) + (lane >> 4);   // the unit this lane works out
  float sb = 0.f, sg = 0.f, p1 = 0.f, r2 = 0.f;
  // the next tile on its way while this one is worked on. Step s: units 2 s (lanes 0..15) and 2 s + 1 (lanes
  // 16..31), eight weights per lane; units beyond the last are not fetched (what stands there is not used)
  auto fetch = [&](long long tile) {
    const int left = (int)min((long long)32, p.units - tile * 32);
    const uint4* const src = reinterpret_cast<const uint4*>(p.w + tile * 32 * kLdpGroup) + lane;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(mybuf);
#pragma unroll
    for (int s = 0; s < 16; s++)
      if (2 * s + (lane >> 4) < left)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + s * 512), "l"(src + s * 32) : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
    const long long u = tile * 32 + (mine < left ? mine : 0);
    sb = __ldg(p.sb + u); sg = __ldg(p.sg + u); p1 = __ldg(p.s1 + u); r2 = __ldg(p.s2 + u);
  };
  long long tile = (long long)blockIdx.x * kLdpWarps + warp;
  if (tile >= ntile) return;
  fetch(tile);
  for (; tile < ntile; tile += stride) {
    const long long u0 = tile * 32;
    const int left = (int)min((long long)32, p.units - u0);   // units of this tile
    const bool have = mine < left;
    uint4 v[16];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int s = 0; s < 16; s++) v[s] = mybuf[s * 32];
    // per lane and step: (smallest, minus largest) of its eight weights
    __half2 mm[16];
#pragma unroll
    for (int s = 0; s < 16; s++) {
      const __half2* q = reinterpret_cast<const __half2*>(&v[s]);
      const __half2 mn = __hmin2(__hmin2(q[0], q[1]), __hmin2(q[2], q[3]));
      const __half2 mx = __hneg2(__hmax2(__hmax2(q[0], q[1]), __hmax2(q[2], q[3])));
      mm[s] = __hmin2(__lows2half2(mn, mx), __highs2half2(mn, mx));
    }
    // after this, mm[0] of lane l is that of step l & 15 over its 16 lanes
    auto halve = [&](auto dist) {
      constexpr int d = decltype(dist)::value;
      const bool up = (lane & d) != 0;
#pragma unroll
      for (int s = 0; s < d; s++) {
        const __half2 a = mm[s], b = mm[s + d];   // (values: a choice between elements would put the array in memory)
        const __half2 keep = up ? b : a, send = up ? a : b;
        mm[s] = __hmin2(keep, __shfl_xor_sync(0xffffffffu, send, d));
      }
    };
    halve(std::integral_constant<int, 8>());
    halve(std::integral_constant<int, 4>());
    halve(std::integral_constant<int, 2>());
    halve(std::integral_constant<int, 1>());
    // (as from infinities of either sign: a unit of nothing but NaN has an empty range)
    mm[0] = __hmin2(mm[0], __half2half2(__ushort_as_half((unsigned short)0x7C00)));
    const float wmin = __low2float(mm[0]), wmax = -__high2float(mm[0]);
    const float lo = __fmul_rn(sb, wmin);
    const float hi = __fmul_rn(sg, wmax);
    const float h = __fsub_rn(hi, lo);
    const float rest = __fsub_rn(1.0f, p1);
    const float p2 = __fmul_rn(rest, r2);
    const float p3 = __fmul_rn(rest, __fsub_rn(1.0f, r2));
    const float t1 = __fmul_rn(p1, 0.5f);   // halving rounds like the division by 2 of the definition
    const float t2 = __fadd_rn(t1, __fmul_rn(__fadd_rn(p1, p2), 0.5f));
    const float t3 = __fadd_rn(t2, __fmul_rn(__fadd_rn(p2, p3), 0.5f));
    if (tile + stride < ntile) fetch(tile + stride);   // (every value of this tile has left the buffer)
    const bool ok = h > 0.0f;
    uint32_t c1 = 0x7FFF7FFFu, c2 = 0x7FFF7FFFu, c3 = 0x7FFF7FFFu;   // no weight reaches a NaN: code 0
    if (ok) {
      const int a = ldp_cut(lo, hi, h, t1), b = ldp_cut(lo, hi, h, t2), c = ldp_cut(lo, hi, h, t3);
      // in ascending order (the code only counts them; they are in order already for sigmoids between 0 and 1)
      const int ab = min(a, b), ba = max(a, b);
      c1 = __half_as_ushort(half_of_key(min(ab, c))) * 0x10001u;
      c2 = __half_as_ushort(half_of_key(max(ab, min(ba, c)))) * 0x10001u;
      c3 = __half_as_ushort(half_of_key(max(ba, c))) * 0x10001u;
    }
    if (have) {
      const float w1 = __fmul_rn(__fadd_rn(t1, t2), 0.5f), w2 = __fmul_rn(__fadd_rn(t2, t3), 0.5f);
      float lv[4] = {__fadd_rn(lo, __fmul_rn(h, 0.0f)), __fadd_rn(lo, __fmul_rn(h, w1)), __fadd_rn(lo, __fmul_rn(h, w2)), __fadd_rn(lo, __fmul_rn(h, 1.0f))};
      if (!ok) lv[0] = lv[1] = lv[2] = lv[3] = lo;
      const __half2 l01 = __halves2half2(__float2half_rn(lv[0]), __float2half_rn(lv[1]));
      const __half2 l23 = __halves2half2(__float2half_rn(lv[2]), __float2half_rn(lv[3]));
      p.lut[u0 + mine] = make_uint2(*reinterpret_cast<const uint32_t*>(&l01), *reinterpret_cast<const uint32_t*>(&l23));
    }
    // Codes. Bit 1 is w >= c_2; bit 0 then is w >= c_3 or w >= c_1. Two weights per register; the j-th pair of a
    // vector drops its codes at bits 4 j and 16 + 4 j.
    uint32_t* const dst = p.words + u0 * (kLdpGroup / 16) + (lane & 1) * 16 + (lane >> 1);
    uint32_t even = 0;
#pragma unroll
    for (int s = 0; s < 16; s++) {
      const int from = s | (lane & 16);   // the lane that worked this unit out
      const uint32_t k1 = __shfl_sync(0xffffffffu, c1, from), k2 = __shfl_sync(0xffffffffu, c2, from),
                     k3 = __shfl_sync(0xffffffffu, c3, from);
      const __half2* q = reinterpret_cast<const __half2*>(&v[s]);
      uint32_t acc = 0;
#pragma unroll
      for (int j = 0; j < 4; j++) {
        const uint32_t m2 = __hge2_mask(q[j], *reinterpret_cast<const __half2*>(&k2));
        const uint32_t k13 = (m2 & k3) | (~m2 & k1);
        const uint32_t m1 = __hge2_mask(q[j], *reinterpret_cast<const __half2*>(&k13));
        acc |= m1 & (0x00010001u << (4 * j));
        acc |= m2 & (0x00020002u << (4 * j));
      }
      acc |= acc >> 14;   // the low sixteen bits: the codes of this lane's eight weights
      if (s % 2 == 0) {
        even = acc;
      } else {
        // Two lanes make a word. An even and an odd step are exchanged with the neighbouring lane, so that the even
        // lane stores a word of the one and the odd lane a word of the other: 128 bytes per warp and store.
        const uint32_t r = __byte_perm(even, acc, 0x5410);
        const uint32_t other = __shfl_xor_sync(0xffffffffu, r, 1);
        const int unit = 2 * (s - 1 + (lane & 1)) + (lane >> 4);   // of word lane >> 1 of a step's sixteen
        if (unit < left) dst[(s >> 1) * 32] = __byte_perm(r, other, (lane & 1) ? 0x3276 : 0x5410);
      }
    }
  }
}

}  // namespace rcp
