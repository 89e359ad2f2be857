// Shared device/host helpers of the RCP W2A4 library (sm_100a).
#pragma once
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace rcp {

constexpr int kMaxTokens = 16;   // skinny regime of the GEMV
constexpr int kMaxK = 65536;

// Loads of what the kernel in front may write (activations, their scales and digits, exported layers). Kernels here are
// launched while that one still runs and wait for it with griddepcontrol.wait, so this data is not constant for their
// lifetime. __ldg promises that it is, and the compiler moves such loads in front of the wait: a layer on the results of the
// layer in front of it read those of an earlier pass. An ordinary load stays behind the wait; its latency (some 0.3 us from
// L2 at worst: one token in a chain, 2048x2048 2.77 -> 2.87 us, 4096x4096 3.71 -> 4.05) is what the data costs.
template <typename T>
__device__ __forceinline__ T ld_input(const T* p) { return *p; }

// dot products of four bytes: unsigned or signed bytes of a, signed bytes of b
__device__ __forceinline__ void dp4a_u8s8(int& d, uint32_t a, uint32_t b) {
  asm("dp4a.u32.s32 %0, %1, %2, %0;" : "+r"(d) : "r"(a), "r"(b));
}
__device__ __forceinline__ void dp4a_s8s8(int& d, uint32_t a, uint32_t b) {
  asm("dp4a.s32.s32 %0, %1, %2, %0;" : "+r"(d) : "r"(a), "r"(b));
}

__device__ __forceinline__ int sext4(uint32_t nib) { return (int)((nib ^ 8u) & 0xFu) - 8; }

// y = s * (L0*S0 + L1*S1 + L2*S2 + L3*S3), fp32 arithmetic, integers converted exactly (|S| < 2^24).
__device__ __forceinline__ __half lut_finish(float s, uint2 lut4, int S0, int S1, int S2, int S3) {
  const __half2 l01 = *reinterpret_cast<const __half2*>(&lut4.x);
  const __half2 l23 = *reinterpret_cast<const __half2*>(&lut4.y);
  float acc = __half2float(__low2half(l01)) * (float)S0;
  acc = fmaf(__half2float(__high2half(l01)), (float)S1, acc);
  acc = fmaf(__half2float(__low2half(l23)), (float)S2, acc);
  acc = fmaf(__half2float(__high2half(l23)), (float)S3, acc);
  return __float2half_rn(s * acc);
}

// L0*S0 + L1*S1 + L2*S2 + L3*S3 alone, in the same order and arithmetic.
__device__ __forceinline__ float lut_sum(uint2 lut4, int S0, int S1, int S2, int S3) {
  const __half2 l01 = *reinterpret_cast<const __half2*>(&lut4.x);
  const __half2 l23 = *reinterpret_cast<const __half2*>(&lut4.y);
  float acc = __half2float(__low2half(l01)) * (float)S0;
  acc = fmaf(__half2float(__high2half(l01)), (float)S1, acc);
  acc = fmaf(__half2float(__low2half(l23)), (float)S2, acc);
  acc = fmaf(__half2float(__high2half(l23)), (float)S3, acc);
  return acc;
}

// x / 7 correctly rounded, for finite x >= 0: the product with the rounded reciprocal and one correction by its exact
// remainder (division by a constant after Markstein; compared with the division itself for all 2^31 values of x). The
// quotient is on the critical path of every quantization, and the general division is four times as long.
__device__ __forceinline__ float div_by_7(float x) {
  constexpr float y = 1.0f / 7.0f;
  const float q = __fmul_rn(x, y);
  return __fmaf_rn(__fmaf_rn(-7.0f, q, x), y, q);
}
// What keeps x = amax * clip_ratio finite, where the correction would turn infinity into NaN. The largest rotated magnitude
// is below 6e6 and the smallest above 6e-10 (a multiple of 2^-24 over the root of 8192 at most), so beyond
// kClipRatioCap every scale but zero is infinity in fp16 whatever the ratio is, and the host passes no larger one; the
// warps' maxima are cut off at kAmaxCap, which only an infinite activation reaches. (Cut off where each warp leaves its
// maximum: one minimum more behind the barrier cost 2.5 % at 2048 tokens of 4096, here it is free.)
constexpr float kClipRatioCap = 1e18f, kAmaxCap = 1e20f;

// 1 / s within one unit in the last place
__device__ __forceinline__ float reciprocal_within_ulp(float s) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(s));
  return r;
}

// q[e] = clamp(round-half-even(v[e] / s), -8, 7) for NV values, the quotient being the IEEE fp32
// division the definition asks for, without dividing in the common case. With rinv = 1 / s (correctly
// rounded), t = v * rinv lies within 2^-23 |v / s| of the exact quotient and the IEEE quotient within half
// an ulp of it; clamped to [-8, 7] (rounding and clamping commute: the bounds are integers) the two differ
// by less than 1.7e-6, so they round to the same integer unless t lies that close to a half-integer.
// Only then (and on exact ties) does the warp redo its values with the division itself; the vote keeps
// the warp together. Rounding: adding 1.5 * 2^23 leaves the rounded integer in the low mantissa bits.
// s > 0 and finite. Every lane of the warp must call.
template <int NV>
__device__ __forceinline__ void quantize_int4(const float (&v)[NV], float s, int (&q)[NV]) {
  const float rinv = __frcp_rn(s);
  bool doubt = false;
#pragma unroll
  for (int e = 0; e < NV; e++) {
    const float t = fminf(fmaxf(__fmul_rn(v[e], rinv), -8.f), 7.f);
    const float biased = __fadd_rn(t, 12582912.f);
    q[e] = __float_as_int(biased) - 0x4B400000;
    doubt |= fabsf(__fsub_rn(t, __fsub_rn(biased, 12582912.f))) > 0.499996f;
  }
  if (__any_sync(0xffffffffu, doubt)) {
#pragma unroll
    for (int e = 0; e < NV; e++) q[e] = max(-8, min(7, __float2int_rn(__fdiv_rn(v[e], s))));
  }
}

// One group's term of the group-wise form: L0*S0 + L1*S1 + L2*S2 + L3*S3 in fp32.
__device__ __forceinline__ float lut_dot(uint2 lut4, int S0, int S1, int S2, int S3) {
  const float2 l01 = __half22float2(*reinterpret_cast<const __half2*>(&lut4.x));
  const float2 l23 = __half22float2(*reinterpret_cast<const __half2*>(&lut4.y));
  float acc = l01.x * (float)S0;
  acc = fmaf(l01.y, (float)S1, acc);
  acc = fmaf(l23.x, (float)S2, acc);
  acc = fmaf(l23.y, (float)S3, acc);
  return acc;
}

}  // namespace rcp
