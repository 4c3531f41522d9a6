// Self-validating words through which the one-launch loops exchange codes, scales, partial sums and points.
#pragma once
#include "lpc_device.cuh"

namespace lpc {

// Tagged 64-bit words (payload | tag << 32): relaxed, device scope, one indivisible access each.
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(unsigned long long* p, uint32_t payload, uint32_t tag) {
  const unsigned long long v = (unsigned long long)payload | ((unsigned long long)tag << 32);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ uint32_t word_tag(unsigned long long w) { return (uint32_t)(w >> 32); }
// Two neighbouring tagged words (16-byte aligned) by one vector access: each 64-bit element is still one indivisible
// access that carries its own tag, the pair need not be.
__device__ __forceinline__ void ld_word2(const unsigned long long* p, unsigned long long& w0, unsigned long long& w1) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w0), "=l"(w1) : "l"(p) : "memory");
}
// W words from p on (8 W bytes, up to 32 at a time; p aligned to them): words of one thread that are fetched one by one touch each sector once
// per word.
template <int W>
__device__ __forceinline__ void ld_words(const unsigned long long* p, unsigned long long (&w)[W]) {
  static_assert(W == 1 || W == 2 || W == 4 || W == 8, "whole accesses");
  if constexpr (W == 1) {
    w[0] = ld_word(p);
  } else if constexpr (W == 2) {
    ld_word2(p, w[0], w[1]);
  } else {
#pragma unroll
    for (int i = 0; i < W; i += 4)
      asm volatile("ld.relaxed.gpu.global.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(w[i]), "=l"(w[i + 1]), "=l"(w[i + 2]), "=l"(w[i + 3]) : "l"(p + i) : "memory");
  }
}
__device__ __forceinline__ void st_word2(unsigned long long* p, uint32_t payload0, uint32_t payload1, uint32_t tag) {
  const unsigned long long v0 = (unsigned long long)payload0 | ((unsigned long long)tag << 32);
  const unsigned long long v1 = (unsigned long long)payload1 | ((unsigned long long)tag << 32);
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(v0), "l"(v1) : "memory");
}
// The same kind of word in shared memory: stored into CTA `cta` of the cluster at the address that `slot` has in
// this CTA, read back from this CTA's own shared memory.
__device__ __forceinline__ void st_cluster_word(const unsigned long long* slot, uint32_t cta, uint32_t payload, uint32_t tag) {
  const unsigned long long v = (unsigned long long)payload | ((unsigned long long)tag << 32);
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(slot)), "r"(cta));
  asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(remote), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ld_shared_word(const unsigned long long* slot) {
  unsigned long long v;
  asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(smem_u32(slot)) : "memory");
  return v;
}

__device__ __forceinline__ uint32_t extract_bits(uint64_t lo, uint64_t hi, int pos, int b) {
  uint64_t v;
  if (pos < 64) {
    v = lo >> pos;
    if (pos + b > 64) v |= hi << (64 - pos);
  } else {
    v = hi >> (pos - 64);
  }
  return (uint32_t)v & ((1u << b) - 1u);
}

}  // namespace lpc
