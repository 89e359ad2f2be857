// Fused activation path: block-Hadamard rotation (Appendix A.2, normalized Sylvester matrix) ->
// per-token absmax symmetric int4 quantization -> nibble packing (Section 4.4 tensor formats).
//
// A token is one vector of K elements and the whole job is latency: a thread-block cluster of C
// CTAs (1, 2, 4 or 8) shares it, each CTA whole rotation blocks, every thread 8 consecutive
// elements. The butterfly strides run in ascending order: 1,2,4 inside the thread's registers,
// 8..128 by warp shuffles, 256 and up through the CTA's shared memory in radix-8 passes. (A rotation
// block never spans CTAs: one block over a token of 2048, 4096 or 8192 elements takes a one-CTA kernel
// further down, as do blocks of at most 512 in most cases.) Each butterfly is one fp32 add and one fp32 subtract
// (lower index first), then one fp32 multiply by 1/sqrt(B): the rounding order is fixed, so the int4
// decision is reproducible bit for bit. The token's absmax meets in distributed shared memory.
#pragma once
#include "common.cuh"

namespace rcp {

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// reads a float at the same shared-memory offset in CTA `rank` of the cluster
__device__ __forceinline__ float ld_cluster_f32(const float* local, uint32_t rank) {
  const uint32_t laddr = (uint32_t)__cvta_generic_to_shared(local);
  uint32_t raddr;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(raddr) : "r"(laddr), "r"(rank));
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(raddr) : "memory");
  return v;
}

// Sends `halves` fp16 numbers at x on their way to L2, one 128-byte line per thread of the first ones. For use before the
// wait for the kernel in front: the L2 is where that kernel would write them, so this can fetch nothing stale. (Activations
// that are not in L2 otherwise arrive behind the next GEMV's weights: 8192x28672 at one token 21.5 -> 20.7 us, 10007x4096 at
// three 8.5 -> 8.4, 28672x4096 at sixteen 24.7 -> 24.3.)
__device__ __forceinline__ void prefetch_token(const __half* x, int halves, int tid) {
  if (tid * 64 < halves) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + tid * 64));
}

struct QuantParams {
  const __half* x;
  uint8_t* xq;
  __half* scale;
  int K, B, lgB;
  int unit, nunits;     // the token is shared out over the cluster in units of `unit` elements (a multiple of B and 64)
  int lg_local;         // B > 256: log2 B, the strides that go through shared memory end below it
  float inv_sqrt_b, clip_ratio;
};

// C = CTAs per token (the cluster size; grid = tokens * C)
template <int C>
__global__ void __launch_bounds__(1024) quantize_act_kernel(const QuantParams p) {
  extern __shared__ float sbuf[];   // 8 floats per thread when B > 256
  __shared__ float s_red[32];
  __shared__ float s_amax;
  const int m = blockIdx.x / C;
  const uint32_t rank = blockIdx.x % C;   // == %cluster_ctarank for a cluster of C along x
  const int tid = threadIdx.x, lane = tid & 31;
  const int B = p.B;
  // Launched with programmatic stream serialization: let the next kernel get started, then wait
  // for the kernel before this one, whose output x may be and whose input xq and scale may be.
  asm volatile("griddepcontrol.launch_dependents;");
  prefetch_token(p.x + (size_t)m * p.K + (size_t)p.K / C / 8 * rank * 8, p.K / C, tid);
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // this CTA's slice of the token
  const int u0 = (int)((long long)p.nunits * rank / C), u1 = (int)((long long)p.nunits * (rank + 1) / C);
  const int start = u0 * p.unit, len = (u1 - u0) * p.unit;
  const int base = start + tid * 8;
  const bool mine = tid * 8 < len;
  const __half* xm = p.x + (size_t)m * p.K;

  float v[8];
  if (mine) {
    const uint4 raw = ld_input(reinterpret_cast<const uint4*>(xm + base));
    const __half2* h2 = reinterpret_cast<const __half2*>(&raw);
#pragma unroll
    for (int e = 0; e < 4; e++) {
      const float2 f = __half22float2(h2[e]);
      v[2 * e] = f.x;
      v[2 * e + 1] = f.y;
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; e++) v[e] = 0.f;
  }

  if (B > 1) {
    // strides 1, 2, 4: inside the registers
#pragma unroll
    for (int h = 1; h < 8; h *= 2) {
      if (h < B) {
#pragma unroll
        for (int e = 0; e < 8; e++) {
          if ((e & h) == 0) {
            const float u = v[e], w = v[e + h];
            v[e] = __fadd_rn(u, w);
            v[e + h] = __fsub_rn(u, w);
          }
        }
      }
    }
    // strides 8 .. 128: lane exchanges (element stride 8*d <-> lane distance d)
#pragma unroll
    for (int d = 1; d < 32; d *= 2) {
      if (8 * d < B) {
        const bool upper = (lane & d) != 0;
#pragma unroll
        for (int e = 0; e < 8; e++) {
          const float other = __shfl_xor_sync(0xffffffffu, v[e], d);
          v[e] = upper ? __fsub_rn(other, v[e]) : __fadd_rn(v[e], other);
        }
      }
    }
    if (B > 256) {
      // strides 256 .. B/2: passes of up to three strides (radix 8) through shared
      // memory. A pass over strides s, 2s, .. (r = 2, 4 or 8 of them combined) works on tuples of r
      // elements s apart; the tuple index maps to an element index with shifts only:
      // element = ((tuple >> log2 s) << log2(r s)) | (tuple & (s - 1)), plus j s for the j-th member.
#pragma unroll
      for (int e = 0; e < 8; e++) sbuf[tid * 8 + e] = v[e];
      __syncthreads();
      for (int ls = 8; ls < p.lg_local;) {
        const int lr = min(3, p.lg_local - ls);   // log2 of the radix of this pass
        float w[8];
        int idx[8];
#pragma unroll
        for (int e = 0; e < 8; e++) {
          const int tau = (tid << (3 - lr)) + (e >> lr);   // tuple index over the slice
          const int j = e & ((1 << lr) - 1);
          idx[e] = ((tau >> ls) << (ls + lr)) + (tau & ((1 << ls) - 1)) + (j << ls);
          w[e] = sbuf[idx[e]];
        }
#pragma unroll
        for (int t = 0; t < 3; t++) {
          const int hh = 1 << t;  // tuple-local stride
          if (t < lr) {
#pragma unroll
            for (int e = 0; e < 8; e++) {
              if ((e & hh) == 0) {
                const float u = w[e], z = w[e + hh];
                w[e] = __fadd_rn(u, z);
                w[e + hh] = __fsub_rn(u, z);
              }
            }
          }
        }
#pragma unroll
        for (int e = 0; e < 8; e++) sbuf[idx[e]] = w[e];
        __syncthreads();
        ls += lr;
      }
#pragma unroll
      for (int e = 0; e < 8; e++) v[e] = sbuf[tid * 8 + e];
    }
#pragma unroll
    for (int e = 0; e < 8; e++) v[e] = __fmul_rn(v[e], p.inv_sqrt_b);
  }

  // token-wide absmax: warp, CTA, cluster
  float amax = 0.f;
#pragma unroll
  for (int e = 0; e < 8; e++) amax = fmaxf(amax, fabsf(v[e]));
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
  if (lane == 0) s_red[tid >> 5] = fminf(amax, kAmaxCap);
  __syncthreads();
  if (tid < 32) {
    float a = (tid < (int)((blockDim.x + 31) >> 5)) ? s_red[tid] : 0.f;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, d));
    if (tid == 0) s_amax = a;
  }
  if constexpr (C > 1) {
    cluster_sync_all();   // every CTA's s_amax is written (and every partner read of sbuf is done)
    amax = 0.f;
#pragma unroll
    for (int r = 0; r < C; r++) amax = fmaxf(amax, ld_cluster_f32(&s_amax, r));
    cluster_sync_all();   // nobody leaves while a partner may still read its shared memory
  } else {
    __syncthreads();
    amax = s_amax;
  }

  const float s32 = div_by_7(__fmul_rn(amax, p.clip_ratio));
  const __half s16 = __float2half_rn(s32);
  const float s = __half2float(s16);
  if (rank == 0 && tid == 0) p.scale[m] = s16;

  int q[8];
  if (s != 0.f) {   // the same for the whole cluster; threads beyond the slice hold zeros
    quantize_int4<8>(v, s, q);
  } else {
#pragma unroll
    for (int e = 0; e < 8; e++) q[e] = 0;
  }
  if (mine) {
    uint32_t packed = 0;
#pragma unroll
    for (int e = 0; e < 8; e++) packed |= (uint32_t)(q[e] & 0xF) << (4 * e);
    *reinterpret_cast<uint32_t*>(p.xq + (size_t)m * (p.K / 2) + base / 2) = packed;
  }
}

// ---------------------------------------------------------------------------------------------
// One CTA per token. The cluster kernel above shares a token out to get at its latency; with many tokens (the
// activations of a prompt) most of its threads wait at barriers or for the cluster while little else is resident. Here
// a persistent CTA takes token after token, one thread per word (16 consecutive elements) or two, the next token's
// activations already on their way, several CTAs per SM, so that one computes while another waits. Nothing is full then:
// issue slots and shared-memory pipe are half busy (16 to 23 warp instructions per 32 elements) with the 1024 threads per SM
// that the registers leave, the rest is latency between exchanges and barriers. Fewer instructions shorten it: adds, products and the rounding work on pairs (the two-wide fp32 instructions round each half like the scalar ones)
// and the clamp of the rounding is left out where it cannot act. Same operations on the same operands in the same
// order as above: bit-identical results. 2048 tokens, us before (cluster, or one CTA of 512 threads with four barriers)
// and now, memory floor: K = 4096 27.1, 10.8, 3.3; K = 8192 33.8, 21.4, 6.5; K = 14336 in blocks of 128 78.4, 25.8, 11.4.
// Fewer barriers also make it the faster form for one token (K = 4096: 2.8 -> 1.8 us).

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }   // a - b, rounded once

// the sixteen values of a word, pair i holding elements 2 i and 2 i + 1: the four stages that pair them (strides below B)
__device__ __forceinline__ void butterflies_word(float2 (&a)[8], int B) {
  if (B > 1) {
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const float u = a[i].x, w = a[i].y;
      a[i] = make_float2(__fadd_rn(u, w), __fsub_rn(u, w));
    }
  }
#pragma unroll
  for (int h = 1; h < 8; h *= 2) {
    if (2 * h < B) {
#pragma unroll
      for (int i = 0; i < 8; i++) {
        if ((i & h) == 0) {
          const float2 u = a[i], w = a[i + h];
          a[i] = add2(u, w);
          a[i + h] = sub2(u, w);
        }
      }
    }
  }
}
__device__ __forceinline__ void word_from_halves(uint4 r0, uint4 r1, float2 (&v)[8]) {
  const uint32_t w[8] = {r0.x, r0.y, r0.z, r0.w, r1.x, r1.y, r1.z, r1.w};
#pragma unroll
  for (int i = 0; i < 8; i++) v[i] = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
}
// Eight packed nibbles from the fp32 numbers 1.5 * 2^23 + q: the low four bits of the pattern are q's.
__device__ __forceinline__ uint32_t pack_nibbles(const float2* b) {
  uint32_t e[4], o[4];
#pragma unroll
  for (int i = 0; i < 4; i++) { e[i] = __float_as_uint(b[i].x); o[i] = __float_as_uint(b[i].y); }
  const uint32_t lo = __byte_perm(__byte_perm(e[0], e[1], 0x0040), __byte_perm(e[2], e[3], 0x0040), 0x5410);
  const uint32_t hi = __byte_perm(__byte_perm(o[0], o[1], 0x0040), __byte_perm(o[2], o[3], 0x0040), 0x5410);
  return (lo & 0x0F0F0F0Fu) | ((hi << 4) & 0xF0F0F0F0u);
}
// the largest magnitude of the three, NaN where any of them is one
__device__ __forceinline__ float max3_magnitude_or_nan(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Rounds NP pairs of values over s > 0 to int4, as the fp32 numbers 1.5 * 2^23 + q. `clamped` false (the same for the
// whole warp): the caller knows that |v / s| < 7.5. Then v * (1 / s), rounded to an integer in the same operation,
// differs by less than 1.2e-6 from the IEEE quotient (the reciprocal is within 2^-23 of its own size, the quotient within
// 2^-22), so the two round alike unless the remainder is within 4e-6 of a half; such a warp
// divides (and one that has met a NaN, or an infinity: s is infinite then, and the product a NaN). Every lane of the warp
// must call.
template <int NP>
__device__ __forceinline__ void quantize_pairs(const float2 (&v)[NP], float s, bool clamped, float2 (&b)[NP]) {
  bool redo = clamped;
  if (!clamped) {
    const float rinv = reciprocal_within_ulp(s);
    const float2 r2 = make_float2(rinv, rinv), magic = make_float2(12582912.f, 12582912.f);
    const float2 minus = make_float2(-1.f, -1.f);
    float worst = 0.f;
#pragma unroll
    for (int i = 0; i < NP; i++) {
      b[i] = __ffma2_rn(v[i], r2, magic);
      const float2 rest = __ffma2_rn(v[i], r2, __ffma2_rn(b[i], minus, magic));   // (magic - b: minus the integer, exactly)
      worst = max3_magnitude_or_nan(worst, rest.x, rest.y);
    }
    redo = __any_sync(0xffffffffu, !(worst <= 0.499996f));
  }
  if (redo) {
#pragma unroll
    for (int i = 0; i < NP; i++) {   // (pair by pair: rare, and fewer registers: 2048 tokens of 8064 in blocks of 64 16.4 -> 14.6 us)
      const float t[2] = {v[i].x, v[i].y};
      int q[2];
      quantize_int4<2>(t, s, q);
      b[i] = make_float2(__int_as_float(q[0] + 0x4B400000), __int_as_float(q[1] + 0x4B400000));
    }
  }
}
// The word's sixteen int4 values, packed.
__device__ __forceinline__ uint2 quantize_word(const float2 (&v)[8], float s, bool clamped) {
  float2 b[8];
  quantize_pairs<8>(v, s, clamped, b);
  return make_uint2(pack_nibbles(b), pack_nibbles(b + 4));
}
// |v| <= amax and s = fp16(amax * clip / 7): with clip >= 0.94 and a normal s, |v / s| <= 7 / 0.94 * (1 + 2^-10) < 7.5.
__device__ __forceinline__ bool needs_clamp(float clip_ratio, float s) { return !(clip_ratio >= 0.94f && s >= 6.103515625e-5f); }

// Strides of 16 and up inside a warp whose lanes hold one word each, below B
__device__ __forceinline__ void butterflies_lanes(float2 (&v)[8], int B, int lane) {
#pragma unroll
  for (int d = 1; d < 32; d *= 2) {   // stride 16 d
    if (16 * d < B) {
      // lower lane: mine + other; upper lane: other - mine (one rounding either way)
      const float sign = (lane & d) ? -1.f : 1.f;
      const float2 s2 = make_float2(sign, sign);
#pragma unroll
      for (int i = 0; i < 8; i++) {
        const float2 other = make_float2(__shfl_xor_sync(0xffffffffu, v[i].x, d), __shfl_xor_sync(0xffffffffu, v[i].y, d));
        v[i] = __ffma2_rn(v[i], s2, other);
      }
    }
  }
}

// Rotation blocks of at most 512 elements (or none): a block lies within a warp (strides 16, 32, .. are lane
// exchanges), only the token's absmax crosses warps. R words per thread, blockDim.x * R >= K / 16, at most T_MAX threads. BLOCK: the
// block size where it is known at compile time, 0: p.B.
template <int R, int T_MAX, int BLOCK>
__global__ void __launch_bounds__(T_MAX, 1024 / T_MAX) quantize_act_rows_kernel(const QuantParams p, int M) {
  __shared__ unsigned s_max[2][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  asm volatile("griddepcontrol.launch_dependents;");
  prefetch_token(p.x + (size_t)blockIdx.x * p.K, p.K, tid);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  extern __shared__ __align__(16) uint4 s_next[];   // [R][2][T]: the next token's activations; a thread copies its own
  const int W = p.K / 16, T = blockDim.x, B = BLOCK ? BLOCK : p.B;
  auto fetch = [&](int m) {
    const __half* const src = p.x + (size_t)m * p.K;
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int w = r * T + tid;
      if (w < W) {
        const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_next + 2 * r * T + tid);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src + 16 * w) : "memory");
        asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(dst + 16 * T), "l"(src + 16 * w + 8) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // words beyond the token: zeros, which no copy ever lands on (a store and a later asynchronous copy are not ordered)
#pragma unroll
  for (int r = 0; r < R; r++)
    if (r * T + tid >= W) s_next[2 * r * T + tid] = s_next[(2 * r + 1) * T + tid] = make_uint4(0, 0, 0, 0);
  int par = 0;
  fetch(blockIdx.x);
  for (int m = blockIdx.x; m < M; m += gridDim.x, par ^= 1) {
    float2 v[R][8];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
    for (int r = 0; r < R; r++) word_from_halves(s_next[2 * r * T + tid], s_next[(2 * r + 1) * T + tid], v[r]);
    if (m + (int)gridDim.x < M) fetch(m + gridDim.x);   // (the values above have been read)
    float amax = 0.f;
#pragma unroll
    for (int r = 0; r < R; r++) {
      butterflies_word(v[r], B);
      butterflies_lanes(v[r], B, lane);
      if (B > 1) {
        const float2 f2 = make_float2(p.inv_sqrt_b, p.inv_sqrt_b);
#pragma unroll
        for (int i = 0; i < 8; i++) v[r][i] = __fmul2_rn(v[r][i], f2);
      }
#pragma unroll
      for (int i = 0; i < 8; i++) amax = fmaxf(amax, fmaxf(fabsf(v[r][i].x), fabsf(v[r][i].y)));
    }
    // non-negative floats order like their patterns
    unsigned am = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
    if (lane == 0) s_max[par][warp] = min(am, __float_as_uint(kAmaxCap));
    __syncthreads();   // (the other half of s_max is free: everybody has read it before coming here)
    am = __reduce_max_sync(0xffffffffu, lane < nwarp ? s_max[par][lane] : 0u);
    const __half s16 = __float2half_rn(div_by_7(__fmul_rn(__uint_as_float(am), p.clip_ratio)));
    const float s = __half2float(s16);
    if (tid == 0) p.scale[m] = s16;
    const bool clamped = needs_clamp(p.clip_ratio, s);
    uint2* const dst = reinterpret_cast<uint2*>(p.xq + (size_t)m * (p.K / 2));
#pragma unroll
    for (int r = 0; r < R; r++) {
      const int w = r * T + tid;
      const uint2 packed = s != 0.f ? quantize_word(v[r], s, clamped) : make_uint2(0, 0);   // (s: the same for the CTA)
      if (w < W) dst[w] = packed;
    }
  }
}

// One rotation block over the whole token, NT = K / 16 threads (K = 2048, 4096 or 8192). Strides 1..8 inside the word;
// 16..128 after a transposition inside the warp, 256 by one lane exchange; 512 and up after a transposition across the
// R = NT / 32 warps, every thread taking 16 / R columns of R values; then back to words, the absmax meeting at the same
// barrier: two barriers per token. One buffer serves all of it, element e of word t at e QP + t: outside the cross-warp
// pass, which lies between the barriers, a warp touches only the columns of its own words.
// Storing a word by element and reading sixteen words of one element with four 16-byte loads (no bank conflicts either
// way) replaces a transposition through a buffer of its own: 2048 tokens of 4096 11.5 -> 10.6 us, of 8192 23.1 -> 21.5.
constexpr int kFullRowsThreads = 1024;   // per SM; with 1280 or 1536 the registers spill (4096: 11.8 and 14.5 us)
template <int NT>
__host__ __device__ constexpr size_t full_rows_smem() { return (size_t)16 * (NT + 4) * 4; }

template <int NT>
__global__ void __launch_bounds__(NT, kFullRowsThreads / NT) quantize_act_full_rows_kernel(const QuantParams p, int M) {
  extern __shared__ __align__(16) float qbuf[];   // full_rows_smem<NT>()
  constexpr int R = NT / 32, QP = NT + 4;
  __shared__ unsigned s_max[2][R];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  asm volatile("griddepcontrol.launch_dependents;");
  prefetch_token(p.x + (size_t)blockIdx.x * (NT * 16), NT * 16, tid);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int e1 = lane & 15, hi = lane & 16;
  float4* const own = reinterpret_cast<float4*>(qbuf + e1 * QP + warp * 32 + hi);   // element e1 of the words hi .. hi + 15
  uint4 raw[2];
  auto fetch = [&](int m) {
    const uint4* const src = reinterpret_cast<const uint4*>(p.x + (size_t)m * (NT * 16)) + 2 * tid;
    raw[0] = ld_input(src);
    raw[1] = ld_input(src + 1);
  };
  int par = 0;
  fetch(blockIdx.x);
  for (int m = blockIdx.x; m < M; m += gridDim.x, par ^= 1) {
    float2 v[8];
    word_from_halves(raw[0], raw[1], v);
    butterflies_word(v, 16);   // strides 1..8
#pragma unroll
    for (int i = 0; i < 8; i++) { qbuf[2 * i * QP + tid] = v[i].x; qbuf[(2 * i + 1) * QP + tid] = v[i].y; }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const float4 f = own[j];
      v[2 * j] = make_float2(f.x, f.y);
      v[2 * j + 1] = make_float2(f.z, f.w);
    }
    butterflies_word(v, 16);   // strides 16..128
    {
      const float sign = hi ? -1.f : 1.f;
      const float2 s2 = make_float2(sign, sign);
#pragma unroll
      for (int i = 0; i < 8; i++) {   // stride 256
        const float2 other = make_float2(__shfl_xor_sync(0xffffffffu, v[i].x, 16), __shfl_xor_sync(0xffffffffu, v[i].y, 16));
        v[i] = __ffma2_rn(v[i], s2, other);
      }
    }
#pragma unroll
    for (int j = 0; j < 4; j++) own[j] = make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y);
    __syncthreads();
    float amax = 0.f;
    // element c R + warp: its R words 32 apart (values 2 i and 2 i + 1 of the thread are words 2 i and 2 i + 1 of R)
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const float* const col = qbuf + ((2 * i / R) * R + warp) * QP + lane;
      v[i] = make_float2(col[(2 * i % R) * 32], col[((2 * i + 1) % R) * 32]);
    }
    butterflies_word(v, R);   // strides 512 ..
#pragma unroll
    for (int i = 0; i < 8; i++) {
      v[i] = __fmul2_rn(v[i], make_float2(p.inv_sqrt_b, p.inv_sqrt_b));
      amax = fmaxf(amax, fmaxf(fabsf(v[i].x), fabsf(v[i].y)));
      float* const col = qbuf + ((2 * i / R) * R + warp) * QP + lane;
      col[(2 * i % R) * 32] = v[i].x;
      col[((2 * i + 1) % R) * 32] = v[i].y;
    }
    // the next token: a barrier, the rounding and the stores ahead of its use, and no registers held before (2048 tokens of
    // 4096 10.99 us with the loads at the start of the pass, 10.83 here; of 8192 21.7 and 21.4)
    if (m + (int)gridDim.x < M) fetch(m + gridDim.x);
    unsigned am = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
    if (lane == 0) s_max[par][warp] = min(am, __float_as_uint(kAmaxCap));
    __syncthreads();
    am = __reduce_max_sync(0xffffffffu, s_max[par][lane % R]);
    const __half s16 = __float2half_rn(div_by_7(__fmul_rn(__uint_as_float(am), p.clip_ratio)));
    const float s = __half2float(s16);
    if (tid == 0) p.scale[m] = s16;
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = make_float2(qbuf[2 * i * QP + tid], qbuf[(2 * i + 1) * QP + tid]);
    const uint2 packed = s != 0.f ? quantize_word(v, s, needs_clamp(p.clip_ratio, s)) : make_uint2(0, 0);
    reinterpret_cast<uint2*>(p.xq + (size_t)m * (NT * 8))[tid] = packed;
  }
}

// ---------------------------------------------------------------------------------------------
// The rotation of one token by 512 threads inside another kernel (the GEMV's in-kernel quantizer), latency bound: as few
// barriers as possible and all threads at work. Same operations in the same order as above: bit-identical results.

// One rotation block over the whole token of K = 512 E elements (E = 4, 8 or 16): thread t holds the elements t E ..
// t E + E - 1 on return, rotated and scaled, and the token's absmax is returned (the same bits in every thread). Strides
// below E in registers; the next log2 E after a transposition inside the warp; up to 16 E by lane exchanges; the sixteen
// warps' strides after a transposition across the warps: there a column of sixteen values, one per warp, is shared by
// 16 / E lanes, E values each, and a last lane exchange or two. Two barriers (named barrier 1, 512 threads).
// buf: full_rotate_bytes<E>() bytes, 16-byte aligned; s_amax: 16 words.
//   One buffer for both transpositions (57344x8192 30.8 -> 30.3 us a call, a ring stage more fitting beside it; with one
// for each before): element e of lane l of warp w at e kQP + 32 w + (w / E) kPL + l. The pads make
// every access below free of bank conflicts.
template <int E>
struct FullRotate {
  static constexpr int kPL = 2 * E;             // the lanes that share a column are kPL apart
  static constexpr int kQP = E == 16 ? 516 : E == 8 ? 548 : 552;
  static constexpr size_t kBytes = (size_t)E * kQP * 4;
};
__host__ constexpr size_t full_rotate_bytes(int K) {
  return K == 2048 ? FullRotate<4>::kBytes : K == 4096 ? FullRotate<8>::kBytes : FullRotate<16>::kBytes;
}

// the stages that pair 2 NP register values (strides 1 .. NP)
template <int NP>
__device__ __forceinline__ void butterflies_pairs(float2 (&a)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; i++) {
    const float u = a[i].x, w = a[i].y;
    a[i] = make_float2(__fadd_rn(u, w), __fsub_rn(u, w));
  }
#pragma unroll
  for (int h = 1; h < NP; h *= 2) {
#pragma unroll
    for (int i = 0; i < NP; i++) {
      if ((i & h) == 0) {
        const float2 u = a[i], w = a[i + h];
        a[i] = add2(u, w);
        a[i + h] = sub2(u, w);
      }
    }
  }
}
template <int NP>
__device__ __forceinline__ void butterfly_exchange(float2 (&a)[NP], int d, bool upper) {
  const float sign = upper ? -1.f : 1.f;
  const float2 s2 = make_float2(sign, sign);
#pragma unroll
  for (int i = 0; i < NP; i++) {
    const float2 other = make_float2(__shfl_xor_sync(0xffffffffu, a[i].x, d), __shfl_xor_sync(0xffffffffu, a[i].y, d));
    a[i] = __ffma2_rn(a[i], s2, other);
  }
}

template <int E>
__device__ __forceinline__ float rotate_full_token(const __half* x, float inv_sqrt_b, float* buf, unsigned* s_amax,
                                                   float2 (&v)[E / 2]) {
  using F = FullRotate<E>;
  constexpr int NP = E / 2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* const mine = buf + warp * 32 + (warp / E) * F::kPL + lane;
  const int e1 = lane % E, l1 = lane - e1;   // after the transposition this lane has element e1 of the lanes l1 .. l1 + E - 1
  float4* const own = reinterpret_cast<float4*>(buf + e1 * F::kQP + warp * 32 + (warp / E) * F::kPL + l1);
  {
    uint32_t raw[NP];
    if constexpr (E == 4) {
      const uint2 r = ld_input(reinterpret_cast<const uint2*>(x) + tid);
      raw[0] = r.x; raw[1] = r.y;
    } else {
#pragma unroll
      for (int i = 0; i < E / 8; i++) {
        const uint4 r = ld_input(reinterpret_cast<const uint4*>(x) + tid * (E / 8) + i);
        raw[4 * i] = r.x; raw[4 * i + 1] = r.y; raw[4 * i + 2] = r.z; raw[4 * i + 3] = r.w;
      }
    }
#pragma unroll
    for (int i = 0; i < NP; i++) v[i] = __half22float2(*reinterpret_cast<const __half2*>(&raw[i]));
  }
  butterflies_pairs<NP>(v);   // strides 1 .. E / 2
#pragma unroll
  for (int i = 0; i < NP; i++) { mine[2 * i * F::kQP] = v[i].x; mine[(2 * i + 1) * F::kQP] = v[i].y; }
  __syncwarp();
#pragma unroll
  for (int j = 0; j < E / 4; j++) {
    const float4 f = own[j];
    v[2 * j] = make_float2(f.x, f.y);
    v[2 * j + 1] = make_float2(f.z, f.w);
  }
  butterflies_pairs<NP>(v);   // strides E .. E E / 2
#pragma unroll
  for (int d = E; d < 32; d *= 2) butterfly_exchange<NP>(v, d, (lane & d) != 0);   // .. 16 E
#pragma unroll
  for (int j = 0; j < E / 4; j++) own[j] = make_float4(v[2 * j].x, v[2 * j].y, v[2 * j + 1].x, v[2 * j + 1].y);
  asm volatile("bar.sync 1, 512;" ::: "memory");
  {
    constexpr int kLC = 16 / E;              // warps that share an element's columns, and lanes that share a column
    const int wq = lane / F::kPL;            // this lane: the values of the warps wq E .. wq E + E - 1
    float* const col = buf + (warp / kLC) * F::kQP + wq * (E * 32 + F::kPL) + (warp % kLC) * F::kPL + lane % F::kPL;
#pragma unroll
    for (int i = 0; i < NP; i++) v[i] = make_float2(col[2 * i * 32], col[(2 * i + 1) * 32]);
    butterflies_pairs<NP>(v);
#pragma unroll
    for (int d = F::kPL; d < 32; d *= 2) butterfly_exchange<NP>(v, d, (lane & d) != 0);
    float amax = 0.f;
#pragma unroll
    for (int i = 0; i < NP; i++) {
      v[i] = __fmul2_rn(v[i], make_float2(inv_sqrt_b, inv_sqrt_b));
      amax = fmaxf(amax, fmaxf(fabsf(v[i].x), fabsf(v[i].y)));
      col[2 * i * 32] = v[i].x;
      col[(2 * i + 1) * 32] = v[i].y;
    }
    const unsigned am = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));   // non-negative: ordered like the patterns
    if (lane == 0) s_amax[warp] = min(am, __float_as_uint(kAmaxCap));
  }
  asm volatile("bar.sync 1, 512;" ::: "memory");
#pragma unroll
  for (int i = 0; i < NP; i++) v[i] = make_float2(mine[2 * i * F::kQP], mine[(2 * i + 1) * F::kQP]);
  return __uint_as_float(__reduce_max_sync(0xffffffffu, s_amax[lane & 15]));
}

// Rotation blocks of B <= 512 elements (1: none): thread t takes the words t, t + 512, .. (NR at most) of the token's W;
// words beyond it are zeros. Returns the token's absmax; one barrier.
template <int NR>
__device__ __forceinline__ float rotate_block_token(const __half* x, int W, int B, float inv_sqrt_b, unsigned* s_amax,
                                                    float2 (&v)[NR][8]) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint4 raw[NR][2];
#pragma unroll
  for (int r = 0; r < NR; r++) {
    const int w = r * 512 + tid;
    raw[r][0] = raw[r][1] = make_uint4(0, 0, 0, 0);
    if (w < W) { raw[r][0] = ld_input(reinterpret_cast<const uint4*>(x) + 2 * w); raw[r][1] = ld_input(reinterpret_cast<const uint4*>(x) + 2 * w + 1); }
  }
  float amax = 0.f;
#pragma unroll
  for (int r = 0; r < NR; r++) {
    word_from_halves(raw[r][0], raw[r][1], v[r]);
    if (r * 512 + warp * 32 < W) {   // (whole warps)
      butterflies_word(v[r], B);
      butterflies_lanes(v[r], B, lane);
      if (B > 1) {
#pragma unroll
        for (int i = 0; i < 8; i++) v[r][i] = __fmul2_rn(v[r][i], make_float2(inv_sqrt_b, inv_sqrt_b));
      }
#pragma unroll
      for (int i = 0; i < 8; i++) amax = fmaxf(amax, fmaxf(fabsf(v[r][i].x), fabsf(v[r][i].y)));
    }
  }
  const unsigned am = __reduce_max_sync(0xffffffffu, __float_as_uint(amax));
  if (lane == 0) s_amax[warp] = min(am, __float_as_uint(kAmaxCap));
  asm volatile("bar.sync 1, 512;" ::: "memory");
  return __uint_as_float(__reduce_max_sync(0xffffffffu, s_amax[lane & 15]));
}

}  // namespace rcp
