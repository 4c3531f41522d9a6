// What the quantizer's kernels share: loads of a group of eight values, its statistics, and its packed bits on their way to memory.
#pragma once
#include "lpc_device.cuh"
#include "lpc_kernels.h"

namespace lpc {

// Eight consecutive values u[j..j+8) of (p - q), zero beyond len.  `vec` says 16-byte loads are legal.
__device__ __forceinline__ void load8(const float* __restrict__ p, const float* __restrict__ q, int64_t j,
                                      int64_t len, bool vec, float* v) {
  if (vec && j + 8 <= len) {
    const float4 a = *reinterpret_cast<const float4*>(p + j);
    const float4 c = *reinterpret_cast<const float4*>(p + j + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = c.x; v[5] = c.y; v[6] = c.z; v[7] = c.w;
    if (q) {
      const float4 e = *reinterpret_cast<const float4*>(q + j);
      const float4 f = *reinterpret_cast<const float4*>(q + j + 4);
      v[0] = __fsub_rn(v[0], e.x); v[1] = __fsub_rn(v[1], e.y); v[2] = __fsub_rn(v[2], e.z); v[3] = __fsub_rn(v[3], e.w);
      v[4] = __fsub_rn(v[4], f.x); v[5] = __fsub_rn(v[5], f.y); v[6] = __fsub_rn(v[6], f.z); v[7] = __fsub_rn(v[7], f.w);
    }
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int64_t i = j + e;
      v[e] = (i < len) ? (q ? __fsub_rn(p[i], q[i]) : p[i]) : 0.f;
    }
  }
}

__device__ __forceinline__ bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
__device__ __forceinline__ bool aligned32(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; }

__device__ __forceinline__ float max3_abs(float m, float a, float b) {
  float r;  // a NaN among the operands comes out as NaN, whose bit pattern is above infinity's
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(a), "f"(b));
  return r;
}

// max |u| into mx; with SUMS the tree sums of the eight values and of their squares, as one pair.
template <bool SUMS>
__device__ __forceinline__ f32x2 stats_group8(const f32x2* v, float& mx) {
  f32x2 pr[4];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    float v0, v1;
    unpack2(v[h], v0, v1);
    mx = max3_abs(mx, v0, v1);
    if constexpr (SUMS) {
      float s0, s1;
      unpack2(mul2_rn(v[h], v[h]), s0, s1);
      pr[h] = pack2(add_rn(v0, v1), add_rn(s0, s1));
    }
  }
  if constexpr (SUMS) return add2_rn(add2_rn(pr[0], pr[1]), add2_rn(pr[2], pr[3]));
  else return 0ull;
}

// The warp's tree sums of its four sweeps, by recursive halving (9 shuffles instead of 40): afterwards lane l < 8 holds
// S1 (bit 2 clear) or S2 of sweep 2 * bit 0 + bit 1.
__device__ __forceinline__ float warp_sums4(const f32x2* pr, int lane) {
  const bool u0 = lane & 1, u1 = lane & 2, u2 = lane & 4;
  const f32x2 k0 = add2_rn(u0 ? pr[2] : pr[0], __shfl_xor_sync(0xFFFFFFFFu, u0 ? pr[0] : pr[2], 1));
  const f32x2 k1 = add2_rn(u0 ? pr[3] : pr[1], __shfl_xor_sync(0xFFFFFFFFu, u0 ? pr[1] : pr[3], 1));
  const f32x2 k = add2_rn(u1 ? k1 : k0, __shfl_xor_sync(0xFFFFFFFFu, u1 ? k0 : k1, 2));
  float a, b;
  unpack2(k, a, b);
  float r = add_rn(u2 ? b : a, __shfl_xor_sync(0xFFFFFFFFu, u2 ? a : b, 4));
  r = add_rn(r, __shfl_xor_sync(0xFFFFFFFFu, r, 8));
  return add_rn(r, __shfl_xor_sync(0xFFFFFFFFu, r, 16));
}

__device__ __forceinline__ void push_code(uint64_t& lo, uint64_t& hi, uint32_t code, int b) {  // (hi, lo) = (hi, lo) << b | code
  const uint32_t w0 = (uint32_t)lo, w1 = (uint32_t)(lo >> 32), w2 = (uint32_t)hi, w3 = (uint32_t)(hi >> 32);
  hi = (uint64_t)__funnelshift_l(w1, w2, b) | ((uint64_t)__funnelshift_l(w2, w3, b) << 32);
  lo = (uint64_t)((w0 << b) | code) | ((uint64_t)__funnelshift_l(w0, w1, b) << 32);
}

// The packed bits of a group at a width known at run time, from its scaled values; 2 to 7 bits by the rule of
// quantize_scaled8, wider codes by conversion to an integer.
__device__ __forceinline__ void quantize_scaled8_rt(const float* s, const U4& r, int b, uint64_t& lo, uint64_t& hi) {
  const uint32_t rw[4] = {r.x, r.y, r.z, r.w};
  lo = hi = 0;
  if (b <= 7) {
    const float SC = __int_as_float((127 - b) << 23), HS = (float)((1 << (b - 1)) - 1) * SC;  // 2^-b and hi 2^-b, exact
    const float C = 1.0f - SC - SC / 131072.f, UP = (float)(1 << (16 + b));
#pragma unroll
    for (int h = 3; h >= 0; --h) {
      const float q0 = fma_ru_sat(fma_rd_sat(s[2 * h], -SC, HS), -1.f, C), q1 = fma_ru_sat(fma_rd_sat(s[2 * h + 1], -SC, HS), -1.f, C);
      float t0, t1;
      unpack2(fma2_ru(pack2(q0, q1), pack2(UP, UP), pack2(8388608.f, 8388608.f)), t0, t1);
      const uint32_t x0 = __dp2a_lo(~rw[h], 0x0001u, __float_as_uint(t0)), x1 = __dp2a_lo(~rw[h], 0x0100u, __float_as_uint(t1));
      const uint32_t two = ((x0 >> 16) & 0xFFu) | (((x1 >> 16) & 0xFFu) << b);
      hi = 0;
      lo = (lo << (2 * b)) | two;
    }
  } else {
    const float l = -(float)(1 << (b - 1)), u = (float)((1 << (b - 1)) - 1);
#pragma unroll
    for (int e = 7; e >= 0; --e) {
      const uint32_t A = (uint32_t)__float2int_ru(__fmaf_ru(fminf(fmaxf(s[e], l), u), 65536.f, -0.5f));
      push_code(lo, hi, (A + (65535u + (65536u << (b - 1))) - lane16(r, e)) >> 16, b);
    }
  }
}

// The b bytes of every thread's group to their place in a sweep's 64 b words, of which `words` exist.  16 bits are
// whole words of a thread's own; the others are put together per warp in shared memory (a warp's 32 groups are 8 b whole
// words), two bytes at a time where b is even.
__device__ __forceinline__ void store_any_width(uint32_t* __restrict__ out, int words, uint64_t lo, uint64_t hi, int b, int tid, int lane,
                                                uint8_t* stage) {
  if (b == 16) {
    if (tid * 4 < words) *reinterpret_cast<uint4*>(out + tid * 4) = make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
    return;
  }
  const int warp = tid >> 5;
  uint8_t* mine = stage + warp * 512 + lane * b;
  __syncwarp();  // the words of the sweep before have been read
  if ((b & 1) == 0) {
    uint16_t* m2 = reinterpret_cast<uint16_t*>(mine);
    for (int i = 0; i < b / 2; ++i) m2[i] = (uint16_t)((i < 4) ? (lo >> (16 * i)) : (hi >> (16 * (i - 4))));
  } else {
    for (int i = 0; i < b; ++i) mine[i] = (uint8_t)((i < 8) ? (lo >> (8 * i)) : (hi >> (8 * (i - 8))));
  }
  __syncwarp();
  const uint32_t* st = reinterpret_cast<const uint32_t*>(stage + warp * 512);
  for (int w = lane; w < 8 * b; w += 32)
    if (warp * 8 * b + w < words) out[warp * 8 * b + w] = st[w];
}

template <int BITS>
__device__ __forceinline__ void store_group(uint32_t* __restrict__ ot, int g, int lane, uint64_t lo) {
  if (BITS == 8) {
    *reinterpret_cast<uint2*>(ot + 2 * g) = make_uint2((uint32_t)lo, (uint32_t)(lo >> 32));
  } else if (BITS == 4) {
    ot[g] = (uint32_t)lo;
  } else if (BITS == 2) {
    const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, (uint32_t)lo, 1);
    if ((lane & 1) == 0) ot[g >> 1] = (uint32_t)lo | (next << 16);
  } else if (BITS == 3) {
    // 24 bits per thread: four neighbouring lanes hold three words; lane i < 3 of them builds word i from its own bits
    // and its neighbour's
    const uint32_t mine = (uint32_t)lo, next = __shfl_down_sync(0xFFFFFFFFu, mine, 1);
    const int i = lane & 3;
    if (i < 3) ot[3 * (g >> 2) + i] = (mine >> (8 * i)) | (next << (24 - 8 * i));
  } else {
    const uint32_t mine = (uint32_t)lo;
    const uint32_t n1 = __shfl_down_sync(0xFFFFFFFFu, mine, 1);
    const uint32_t n2 = __shfl_down_sync(0xFFFFFFFFu, mine, 2);
    const uint32_t n3 = __shfl_down_sync(0xFFFFFFFFu, mine, 3);
    if ((lane & 3) == 0) ot[g >> 2] = mine | (n1 << 8) | (n2 << 16) | (n3 << 24);
  }
}

// A group's packed bits at group g of the segment; words from `words` on do not exist.
template <int BITS>
__device__ __forceinline__ void store_group_bounded(uint32_t* __restrict__ out, int g, int lane, uint64_t lo, int words) {
  if (BITS == 8) {
    if (2 * g < words) *reinterpret_cast<uint2*>(out + 2 * g) = make_uint2((uint32_t)lo, (uint32_t)(lo >> 32));
  } else if (BITS == 4) {
    if (g < words) out[g] = (uint32_t)lo;
  } else if (BITS == 2) {
    const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, (uint32_t)lo, 1);
    if ((lane & 1) == 0 && (g >> 1) < words) out[g >> 1] = (uint32_t)lo | (next << 16);
  } else if (BITS == 3) {
    const uint32_t mine = (uint32_t)lo, next = __shfl_down_sync(0xFFFFFFFFu, mine, 1);
    const int i = lane & 3, w = 3 * (g >> 2) + i;
    if (i < 3 && w < words) out[w] = (mine >> (8 * i)) | (next << (24 - 8 * i));
  } else {
    const uint32_t mine = (uint32_t)lo;
    const uint32_t n1 = __shfl_down_sync(0xFFFFFFFFu, mine, 1);
    const uint32_t n2 = __shfl_down_sync(0xFFFFFFFFu, mine, 2);
    const uint32_t n3 = __shfl_down_sync(0xFFFFFFFFu, mine, 3);
    if ((lane & 3) == 0 && (g >> 2) < words) out[g >> 2] = mine | (n1 << 8) | (n2 << 16) | (n3 << 24);
  }
}

}  // namespace lpc
