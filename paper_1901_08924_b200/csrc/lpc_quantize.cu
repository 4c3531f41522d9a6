// Quantization step of Algorithm 1 (step 7) for stand-alone worker vectors: the scale of Eq. 2
// (a reduction pass), then the stochastic quantizer Q_(delta,b) of Section 2.2 and bit packing
// (a second pass).  Vectors may be split into tensor segments that each get their own scale.
//
// Layout of the work: a CTA owns one tile of TILE consecutive coordinates of one segment of one
// worker; a thread owns groups of 8 consecutive coordinates (two 128-bit loads, one Philox block,
// 8*b packed bits).  All sums follow the balanced binary tree over the coordinate index, so the
// scale -- and with it every code -- does not depend on the tiling.
#include <cooperative_groups.h>

#include <type_traits>

#include "lpc_quantize.cuh"

namespace lpc {
namespace {

constexpr int QT = 256;                   // threads per CTA
constexpr int QGROUP = QT * 8;            // coordinates per CTA sweep
constexpr int QITER = TILE / QGROUP;      // sweeps per tile
static_assert(QITER * QGROUP == TILE, "tile must be a whole number of sweeps");

// Eight whole values as four pairs: one 32-byte load where the alignment allows it, two 16-byte loads through L1
// otherwise (without L1 each of them would fetch the whole sector).  LAST: nobody reads them again, L2 may drop them.
template <bool LAST>
__device__ __forceinline__ void load8v(const float* p, bool al32, f32x2* v) {
  if (al32) {
    if constexpr (LAST)
      asm volatile("ld.global.L1::no_allocate.L2::evict_first.v4.b64 {%0, %1, %2, %3}, [%4];"
                   : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
    else
      asm volatile("ld.global.L1::no_allocate.v4.b64 {%0, %1, %2, %3}, [%4];"
                   : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
  } else {
    asm volatile("ld.global.v2.b64 {%0, %1}, [%4];\n\tld.global.v2.b64 {%2, %3}, [%4+16];"
                 : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p));
  }
}

// The same with a cache policy of L2 that is chosen at run time.
__device__ __forceinline__ void load8v_policy(const float* p, bool al32, uint64_t policy, f32x2* v) {
  if (al32)
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.b64 {%0, %1, %2, %3}, [%4], %5;"
                 : "=l"(v[0]), "=l"(v[1]), "=l"(v[2]), "=l"(v[3]) : "l"(p), "l"(policy));
  else
    load8v<false>(p, false, v);
}

// ---- pass 1: per-tile partial (max |u| as bit pattern, tree sums of u and u^2) ---------------------------
// Bound by memory: all of a thread's loads of a tile are under way before the first is used, and the sums of the four
// sweeps share their shuffles.  POLICY: the loads carry a cache policy.
template <bool NEED_SUMS, bool POLICY>
__device__ __forceinline__ void stats_tile(const QuantArgs& a, int tile, int worker, uint64_t policy, float* sh1, float* sh2, uint32_t* shm) {
  auto load = [&](const float* from, bool al32, f32x2* v) {
    if constexpr (POLICY) load8v_policy(from, al32, policy, v);
    else load8v<false>(from, al32, v);
  };
  const int seg = a.tile_seg ? a.tile_seg[tile] : 0;
  const SegInfo s = a.segs[seg];
  const int64_t tstart = (int64_t)(tile - s.tile_first) * TILE;
  const float* p = a.U + (int64_t)worker * a.ld + s.off;
  const float* q = a.U_sub ? a.U_sub + (int64_t)worker * a.ld + s.off : nullptr;
  const bool vec = aligned16(p) && (!q || aligned16(q)), al32 = aligned32(p) && (!q || aligned32(q));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  float mx = 0.f;
  f32x2 pr[QITER];
  if (vec && tstart + TILE <= s.len) {
    const float* pt = p + tstart + tid * 8;
    if (!q) {
      f32x2 v[QITER][4];
#pragma unroll
      for (int it = 0; it < QITER; ++it) load(pt + it * QGROUP, al32, v[it]);
#pragma unroll
      for (int it = 0; it < QITER; ++it) pr[it] = stats_group8<NEED_SUMS>(v[it], mx);
    } else {
      const float* qt = q + tstart + tid * 8;
#pragma unroll
      for (int half = 0; half < QITER; half += 2) {
        f32x2 v[2][4], w[2][4];
#pragma unroll
        for (int it = 0; it < 2; ++it) {
          load(pt + (half + it) * QGROUP, al32, v[it]);
          load(qt + (half + it) * QGROUP, al32, w[it]);
        }
#pragma unroll
        for (int it = 0; it < 2; ++it) {
#pragma unroll
          for (int h = 0; h < 4; ++h) v[it][h] = sub2_rn(v[it][h], w[it][h]);
          pr[half + it] = stats_group8<NEED_SUMS>(v[it], mx);
        }
      }
    }
  } else {
#pragma unroll
    for (int it = 0; it < QITER; ++it) {
      float u[8];
      load8(p, q, tstart + (int64_t)it * QGROUP + tid * 8, s.len, vec, u);
      const f32x2 u2[4] = {pack2(u[0], u[1]), pack2(u[2], u[3]), pack2(u[4], u[5]), pack2(u[6], u[7])};
      pr[it] = stats_group8<NEED_SUMS>(u2, mx);
    }
  }
  const uint32_t wm = warp_max_u32(__float_as_uint(mx) & 0x7FFFFFFFu);
  if (lane == 0) shm[warp] = wm;
  if (NEED_SUMS) {
    const float r = warp_sums4(pr, lane);
    const int j = (((lane & 1) * 2) + ((lane >> 1) & 1)) * 8 + warp;
    if (lane < 4) sh1[j] = r;
    else if (lane < 8) sh2[j] = r;
  }
  __syncthreads();
  const int64_t o = (int64_t)worker * a.ntiles + tile;
  if (warp == 0) {
    const uint32_t m = warp_max_u32(shm[lane & 7]);
    const float r = NEED_SUMS ? warp_tree_sum(sh1[lane]) : 0.f;
    if (lane == 0) {
      a.pmax[o] = m;
      if (NEED_SUMS) a.ps1[o] = r;
    }
  } else if (NEED_SUMS && warp == 1) {
    const float r = warp_tree_sum(sh2[lane]);
    if (lane == 0) a.ps2[o] = r;
  }
}

// POLICY: the second pass goes back from the end, so the tiles worth keeping in L2 are the last `keep` ones: those before them
// are read so that they go first.
template <bool NEED_SUMS, bool POLICY>
__global__ void __launch_bounds__(QT) stats_kernel(QuantArgs a, int keep) {
  launch_dependents();
  wait_for_launch_before();
  __shared__ float sh1[QITER * 8], sh2[QITER * 8];
  __shared__ uint32_t shm[8];
  uint64_t policy = 0;
  if constexpr (POLICY) {
    if ((int64_t)blockIdx.y * a.ntiles + blockIdx.x < (int64_t)a.N * a.ntiles - keep)
      asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
    else
      asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(policy));
  }
  stats_tile<NEED_SUMS, POLICY>(a, blockIdx.x, blockIdx.y, policy, sh1, sh2, shm);
}

// Tree sums over `count` tile partials of both kinds by one CTA of QT threads (leaf order = tile order): a thread owns a
// power-of-two stretch of leaves, eight loads of either array in flight.
__device__ __forceinline__ void block_tree_sums(const float* __restrict__ v1, const float* __restrict__ v2, int count,
                                                float* sh16, float& S1, float& S2) {
  int P = 1;
  while (P < count) P <<= 1;
  const int chunk = (P >= QT) ? P / QT : 1;
  const int lo = threadIdx.x * chunk;
  float a = 0.f, b = 0.f;
  if (chunk < 8) {
    float x[4], y[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // written by other CTAs: read where they wrote it
      const bool in = i < chunk && lo + i < count;
      x[i] = in ? __ldcg(v1 + lo + i) : 0.f;
      y[i] = in ? __ldcg(v2 + lo + i) : 0.f;
    }
    if (chunk == 1) { a = x[0]; b = y[0]; }
    else if (chunk == 2) { a = add_rn(x[0], x[1]); b = add_rn(y[0], y[1]); }
    else { a = tree4(x[0], x[1], x[2], x[3]); b = tree4(y[0], y[1], y[2], y[3]); }
  } else {
    float st1[24], st2[24];  // one pending sum per level
    int top = 0;
    for (int i = 0; i < chunk; i += 8) {
      float x[8], y[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const bool in = lo + i + e < count;
        x[e] = in ? __ldcg(v1 + lo + i + e) : 0.f;
        y[e] = in ? __ldcg(v2 + lo + i + e) : 0.f;
      }
      a = tree8(x);
      b = tree8(y);
      for (int idx = i >> 3; idx & 1; idx >>= 1) {
        --top;
        a = add_rn(st1[top], a);
        b = add_rn(st2[top], b);
      }
      st1[top] = a;
      st2[top] = b;
      ++top;
    }
  }
  a = warp_tree_sum(a);
  b = warp_tree_sum(b);
  if ((threadIdx.x & 31) == 0) { sh16[threadIdx.x >> 5] = a; sh16[8 + (threadIdx.x >> 5)] = b; }
  __syncthreads();
  S1 = tree8(sh16);
  S2 = tree8(sh16 + 8);
}

// ---- between the passes: Eq. 2 from the tile partials --------------------------------------------------------------
// The scale record of (segment, worker), the scale for the caller and the cleared count; one thread.
__device__ __forceinline__ void write_scale(const QuantArgs& a, const SegInfo& s, int seg, int worker, uint32_t m, float S1, float S2) {
  const Scale sc = make_scale(m, S1, S2, s.len, a.b, a.clip_mode, a.clip_value);
  ScaleRec r;
  r.delta = sc.delta; r.rdelta = sc.rdelta; r.T = sc.T; r.lower = sc.lower; r.flags = sc.flags;
  r.pad0 = r.pad1 = r.pad2 = 0;
  // the threshold is the largest magnitude: nothing can lie outside the hull, and nothing has to be counted
  if (sc.T >= __uint_as_float(m) && (!a.shared_scale || a.clip_mode == CLIP_NONE)) r.flags |= SCALE_NONE_OUTSIDE;
  const int64_t o = (int64_t)worker * a.nseg + seg;
  a.scales[o] = r;
  a.delta_out[o] = r.delta;
  a.clipped_out[o] = 0;
  if (r.flags & 2u) atomicOr(a.dev_status, DEV_NONFINITE);
}

// One CTA per (segment, worker); also covers segments without a single coordinate.
__global__ void __launch_bounds__(QT) finish_kernel(QuantArgs a) {
  launch_dependents();
  wait_for_launch_before();
  __shared__ float sh16[16];
  __shared__ uint32_t shm[8];
  const int seg = blockIdx.x, worker = blockIdx.y;
  const SegInfo s = a.segs[seg];
  const int64_t base = (int64_t)worker * a.ntiles + s.tile_first;
  uint32_t mx = 0;
#pragma unroll 8
  for (int t = threadIdx.x; t < s.tile_count; t += QT) mx = max(mx, __ldcg(a.pmax + base + t));
  mx = warp_max_u32(mx);
  if ((threadIdx.x & 31) == 0) shm[threadIdx.x >> 5] = mx;
  float S1 = 0.f, S2 = 0.f;
  if (a.clip_mode == CLIP_STD) block_tree_sums(a.ps1 + base, a.ps2 + base, s.tile_count, sh16, S1, S2);
  else __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t m = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) m = max(m, shm[w]);
    write_scale(a, s, seg, worker, m, S1, S2);
  }
}

// ---- schemes (b), (c) of Section 3.2: delta_t = max_i delta_t^i.  delta^i = T^i / levels grows with the threshold
// T^i, so the record of the worker with the largest threshold is the unified scale; it replaces every worker's
// record of the segment.  Workers whose own vector is zero then send zeros on the shared grid; when every worker
// is degenerate nothing changes.  One warp per segment.
__global__ void __launch_bounds__(32) share_scale_kernel(QuantArgs a) {
  launch_dependents();
  wait_for_launch_before();
  const int seg = blockIdx.x, lane = threadIdx.x;
  float bestT = -1.f;
  int best = -1;
  for (int i = lane; i < a.N; i += 32) {
    const ScaleRec r = a.scales[(int64_t)i * a.nseg + seg];
    if (!(r.flags & 1u) && r.T > bestT) { bestT = r.T; best = i; }  // the first worker among equal thresholds
  }
#pragma unroll
  for (int m = 16; m >= 1; m >>= 1) {
    const float oT = __shfl_xor_sync(0xFFFFFFFFu, bestT, m);
    const int ob = __shfl_xor_sync(0xFFFFFFFFu, best, m);
    if (ob >= 0 && (best < 0 || oT > bestT || (oT == bestT && ob < best))) { bestT = oT; best = ob; }
  }
  if (best < 0) return;
  const ScaleRec r = a.scales[(int64_t)best * a.nseg + seg];
  __syncwarp();
  for (int i = lane; i < a.N; i += 32) {
    a.scales[(int64_t)i * a.nseg + seg] = r;
    a.delta_out[(int64_t)i * a.nseg + seg] = r.delta;
  }
}

// ---- pass 2: quantize and pack -----------------------------------------------------------------------------
// BITS = 1, 2, 3, 4, 8: register/shuffle packing with direct coalesced stores.
// BITS = 0: any b in 1..16 read from the arguments; each thread's 8*b bits are b whole bytes, staged
//           through shared memory and written out as words.
// A CTA takes a run of up to QRUN consecutive tiles of one worker.  Runs that consist of whole tiles of one segment of
// 16-byte aligned vectors (all but a segment's last tiles) go through a software-pipelined loop: nothing is tested per
// group and every index is a small offset from the run's base.  Everything else goes tile by tile through the general code.
// Runs are handed out from the last worker's last tile back: the values that the first pass read last (up to some 80 MB)
// are still in L2.
constexpr int QRUN = 8;

// One atomic addition per CTA to a message's count (all threads call this with their own part).  With one per warp and tile,
// 131,072 additions to eight neighbouring words took 8 x 2^24 values at b = 32 from 240 to 378 us.
__device__ __forceinline__ void add_count(uint32_t n, uint32_t* dst) {
  __shared__ uint32_t part[QT / 32];
  n = __reduce_add_sync(0xFFFFFFFFu, n);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
#pragma unroll
    for (int w = 0; w < QT / 32; ++w) t += part[w];
    if (t) atomicAdd(dst, t);
  }
}

// `nsweeps` sweeps (a multiple of 4) of QGROUP coordinates from pt/qt (this thread's first group); HAS_Q: u = p - q.
// 64 bytes per thread are in flight while a group is quantized: a group's registers are loaded again as soon as its
// values have been scaled and counted.
template <int BITS, bool COUNT, bool HAS_Q>
__device__ __forceinline__ void quantize_run(const QuantArgs& a, const ScaleRec& sc, const float* __restrict__ pt,
                                             const float* __restrict__ qt, bool al32, uint32_t block0,
                                             uint32_t* __restrict__ ot, int nsweeps, int worker, int tid, int lane, float& fclip,
                                             uint8_t* stage) {
  float s[8];
  f32x2 v0[4], v1[4];
  auto finish = [&](int sweep) {
    const int g = sweep * (QGROUP / 8) + tid;  // coordinate group inside the run
    const U4 r = stream_block(a.seed, TAG_ROUND, (uint32_t)worker, a.k, block0 + (uint32_t)g);
    if constexpr (BITS != 0) {
      store_group<BITS>(ot, g, lane, quantize_scaled8<BITS ? BITS : 1>(s, r));
    } else {
      uint64_t lo, hi;
      quantize_scaled8_rt(s, r, a.b, lo, hi);
      store_any_width(ot + (int64_t)sweep * (QGROUP / 32) * a.b, (QGROUP / 32) * a.b, lo, hi, a.b, tid, lane, stage);
    }
  };
  load8v<true>(pt, al32, v0);
  load8v<true>(HAS_Q ? qt : pt + QGROUP, al32, v1);
  if constexpr (HAS_Q) {
#pragma unroll 1
    for (int sweep = 0; sweep < nsweeps; ++sweep) {
#pragma unroll
      for (int h = 0; h < 4; ++h) v0[h] = sub2_rn(v0[h], v1[h]);
      scale_group8<COUNT>(v0, sc.rdelta, sc.T, sc.lower, fclip, s);
      if (sweep + 1 < nsweeps) {
        load8v<true>(pt + (sweep + 1) * QGROUP, al32, v0);
        load8v<true>(qt + (sweep + 1) * QGROUP, al32, v1);
      }
      finish(sweep);
    }
  } else {
#pragma unroll 1
    for (int sweep = 0; sweep < nsweeps; sweep += 2) {
      scale_group8<COUNT>(v0, sc.rdelta, sc.T, sc.lower, fclip, s);
      if (sweep + 2 < nsweeps) load8v<true>(pt + (sweep + 2) * QGROUP, al32, v0);
      finish(sweep);
      scale_group8<COUNT>(v1, sc.rdelta, sc.T, sc.lower, fclip, s);
      if (sweep + 2 < nsweeps) load8v<true>(pt + (sweep + 3) * QGROUP, al32, v1);
      finish(sweep + 1);
    }
  }
}

template <int BITS, bool COUNT>
__device__ __forceinline__ void quantize_tile(const QuantArgs& a, int tile, int worker, uint8_t* stage, const ScaleRec& sc) {
  const int seg = a.tile_seg ? a.tile_seg[tile] : 0;
  const SegInfo s = a.segs[seg];
  const int64_t tstart = (int64_t)(tile - s.tile_first) * TILE;
  const float* p = a.U + (int64_t)worker * a.ld + s.off;
  const float* q = a.U_sub ? a.U_sub + (int64_t)worker * a.ld + s.off : nullptr;
  const bool vec = aligned16(p) && (!q || aligned16(q));
  const int tid = threadIdx.x, lane = tid & 31;
  const int b = BITS ? BITS : a.b;
  const bool degenerate = (sc.flags & 1u) != 0;
  const uint32_t zero_code = (b == 1) ? 0u : (1u << (b - 1));
  uint32_t* out = a.codes + (int64_t)worker * a.stride_words + s.word_off;

  uint32_t nclip = 0;
  float fclip = 0.f;
#pragma unroll
  for (int it = 0; it < QITER; ++it) {
    const int64_t sweep0 = tstart + (int64_t)it * QGROUP;  // first coordinate of this sweep (segment-local)
    const int64_t j = sweep0 + tid * 8;
    uint64_t lo = 0, hi = 0;  // this thread's 8*b bits
    const int nvalid = (j < s.len) ? (int)min((int64_t)8, s.len - j) : 0;
    if (nvalid > 0) {
      float v[8];
      load8(p, q, j, s.len, vec, v);
      if (!degenerate) {
        const U4 r = stream_block(a.seed, TAG_ROUND, (uint32_t)worker, a.k, s.block_base + (uint32_t)(j >> 3));
        if constexpr (BITS != 0) {
          // all eight coordinates are computed without bounds tests (zero padding is inside the hull and is
          // never counted); codes past the end are masked off below
          lo = quantize_group8<BITS ? BITS : 1, COUNT>(v, sc.rdelta, r, sc.T, sc.lower, fclip);
          if (nvalid < 8) lo &= (1ull << (nvalid * BITS)) - 1ull;
        } else {
#pragma unroll
          for (int e = 7; e >= 0; --e) {  // from the last code down, everything so far moves up by one code
            uint32_t code = quantize_code_rt(v[e], sc.rdelta, lane16(r, e), b);
            if (e >= nvalid) code = 0u;
            else if (COUNT) nclip += (v[e] > sc.T || v[e] < sc.lower) ? 1u : 0u;
            push_code(lo, hi, code, b);
          }
        }
      } else {
        for (int e = 0; e < nvalid; ++e) {
          const int pos = e * b;
          if (pos < 64) {
            lo |= (uint64_t)zero_code << pos;
            if (pos + b > 64) hi |= (uint64_t)zero_code >> (64 - pos);
          } else {
            hi |= (uint64_t)zero_code << (pos - 64);
          }
        }
      }
    }
    // ---- store
    if (BITS == 8) {
      const int64_t w = (j >> 3) * 2;
      if (w < s.pad_words) *reinterpret_cast<uint2*>(out + w) = make_uint2((uint32_t)lo, (uint32_t)(lo >> 32));
    } else if (BITS == 4) {
      const int64_t w = j >> 3;
      if (w < s.pad_words) out[w] = (uint32_t)lo;
    } else if (BITS == 2) {
      const uint32_t mine = (uint32_t)lo;  // 16 bits
      const uint32_t next = __shfl_down_sync(0xFFFFFFFFu, mine, 1);
      const int64_t w = j >> 4;
      if ((lane & 1) == 0 && w < s.pad_words) out[w] = mine | (next << 16);
    } else if (BITS == 1) {
      const uint32_t mine = (uint32_t)lo;  // 8 bits
      const uint32_t n1 = __shfl_down_sync(0xFFFFFFFFu, mine, 1);
      const uint32_t n2 = __shfl_down_sync(0xFFFFFFFFu, mine, 2);
      const uint32_t n3 = __shfl_down_sync(0xFFFFFFFFu, mine, 3);
      const int64_t w = j >> 5;
      if ((lane & 3) == 0 && w < s.pad_words) out[w] = mine | (n1 << 8) | (n2 << 16) | (n3 << 24);
    } else if (BITS == 3) {
      const uint32_t mine = (uint32_t)lo, next = __shfl_down_sync(0xFFFFFFFFu, mine, 1);  // 24 bits each
      const int i = lane & 3;
      const int64_t w = 3 * (j >> 5) + i;
      if (i < 3 && w < s.pad_words) out[w] = (mine >> (8 * i)) | (next << (24 - 8 * i));
    } else {
      store_any_width(out + (sweep0 >> 5) * b, (int)min((int64_t)(QGROUP / 32) * b, s.pad_words - (sweep0 >> 5) * b), lo, hi, b, tid, lane, stage);
    }
  }
  nclip = __reduce_add_sync(0xFFFFFFFFu, nclip + (uint32_t)fclip);
  if (COUNT && lane == 0 && nclip) atomicAdd(&a.clipped_out[(int64_t)worker * a.nseg + seg], nclip);
}

// The run [tile, tile + whole) of whole tiles of one segment, by all threads of the CTA.
template <int BITS, bool COUNT>
__device__ __forceinline__ void quantize_whole_tiles(const QuantArgs& a, const SegInfo& s, const ScaleRec& sc, const float* p, const float* q,
                                                     int tile, int whole, int seg, int worker, uint8_t* stage) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t tstart = (int64_t)(tile - s.tile_first) * TILE;
  const uint32_t block0 = s.block_base + (uint32_t)(tstart >> 3);
  uint32_t* ot = a.codes + (int64_t)worker * a.stride_words + s.word_off + (tstart >> 5) * (BITS ? BITS : a.b);
  const bool al32 = aligned32(p) && (!q || aligned32(q));
  const float* pt = p + tstart + tid * 8;
  float fclip = 0.f;
  if (q) {
    const float* qt = q + tstart + tid * 8;
    if (COUNT && !(sc.flags & SCALE_NONE_OUTSIDE))
      quantize_run<BITS, true, true>(a, sc, pt, qt, al32, block0, ot, whole * QITER, worker, tid, lane, fclip, stage);
    else
      quantize_run<BITS, false, true>(a, sc, pt, qt, al32, block0, ot, whole * QITER, worker, tid, lane, fclip, stage);
  } else {
    if (COUNT && !(sc.flags & SCALE_NONE_OUTSIDE))
      quantize_run<BITS, true, false>(a, sc, pt, nullptr, al32, block0, ot, whole * QITER, worker, tid, lane, fclip, stage);
    else
      quantize_run<BITS, false, false>(a, sc, pt, nullptr, al32, block0, ot, whole * QITER, worker, tid, lane, fclip, stage);
  }
  if (COUNT && !(sc.flags & SCALE_NONE_OUTSIDE)) add_count((uint32_t)fclip, &a.clipped_out[(int64_t)worker * a.nseg + seg]);
}

template <int BITS, bool COUNT>
__global__ void __launch_bounds__(QT, 4) quantize_kernel(QuantArgs a, int run) {
  launch_dependents();
  wait_for_launch_before();
  const int worker = (int)(gridDim.y - 1 - blockIdx.y);
  const int tile0 = (int)(gridDim.x - 1 - blockIdx.x) * run;
  const int ntl = min(run, a.ntiles - tile0);
  __shared__ __align__(16) uint8_t stage[BITS == 0 ? QT * 16 : 16];
  {
    const int seg = a.tile_seg ? a.tile_seg[tile0] : 0;
    const int seg_last = a.tile_seg ? a.tile_seg[tile0 + ntl - 1] : 0;  // tiles are numbered segment by segment
    if (seg == seg_last) {
      const SegInfo s = a.segs[seg];
      const float* p = a.U + (int64_t)worker * a.ld + s.off;
      const float* q = a.U_sub ? a.U_sub + (int64_t)worker * a.ld + s.off : nullptr;
      const ScaleRec sc = a.scales[(int64_t)worker * a.nseg + seg];
      if (aligned16(p) && (!q || aligned16(q)) && !(sc.flags & 1u) && (int64_t)(tile0 + ntl - s.tile_first) * TILE <= s.len) {
        quantize_whole_tiles<BITS, COUNT>(a, s, sc, p, q, tile0, ntl, seg, worker, stage);
        return;
      }
    }
  }
  for (int t = 0; t < ntl; ++t) {
    if (BITS == 0 && t > 0) __syncthreads();  // the staging buffer is reused from tile to tile
    const int seg = a.tile_seg ? a.tile_seg[tile0 + t] : 0;
    quantize_tile<BITS, COUNT>(a, tile0 + t, worker, stage, a.scales[(int64_t)worker * a.nseg + seg]);
  }
}

// ---- one cluster per worker for vectors of at most 8 tiles ----------------------------------------------------------
// A CTA holds its tile in registers from the statistics to the codes; the tile partials go to all CTAs of the cluster
// through distributed shared memory and every CTA forms the scale itself (same partials, same tree, same bits).  Nothing
// is looked at twice, no counter is kept, and the launch is a plain one: a call of 4 x 1,000 values takes 4.6 us of host
// time and one pass over the tile, against 8.2 us for a cooperative launch with its grid-wide hand-over.
constexpr int CTILES = 8;
struct ClusterSmem {
  float s1[QITER * 8], s2[QITER * 8];
  uint32_t mx[8], clip[8];
  float p1[CTILES], p2[CTILES];       // the tiles' partials, written by all CTAs of the cluster
  uint32_t pmx[CTILES], pclip[CTILES];
  ScaleRec sc;
};

template <int BITS, bool NEED_SUMS>
__global__ void __launch_bounds__(QT) quantize_cluster_kernel(QuantArgs a) {
  __shared__ ClusterSmem sm;
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster.block_rank(), ctas = (int)cluster.num_blocks(), worker = blockIdx.y;
  const SegInfo s = a.segs[0];
  const float* p = a.U + (int64_t)worker * a.ld;
  const float* q = a.U_sub ? a.U_sub + (int64_t)worker * a.ld : nullptr;
  const bool vec = aligned16(p) && (!q || aligned16(q)), al32 = aligned32(p);
  const int len = (int)s.len, j0 = rank * TILE + tid * 8;
  wait_for_launch_before();

  f32x2 v[QITER][4], pr[QITER];
  float mx = 0.f;
  if (vec && !q && (rank + 1) * TILE <= len) {
#pragma unroll
    for (int it = 0; it < QITER; ++it) load8v<false>(p + j0 + it * QGROUP, al32, v[it]);
  } else {
#pragma unroll
    for (int it = 0; it < QITER; ++it) {
      float u[8];
      load8(p, q, j0 + it * QGROUP, len, vec, u);
#pragma unroll
      for (int h = 0; h < 4; ++h) v[it][h] = pack2(u[2 * h], u[2 * h + 1]);
    }
  }
#pragma unroll
  for (int it = 0; it < QITER; ++it) pr[it] = stats_group8<NEED_SUMS>(v[it], mx);
  const uint32_t wm = warp_max_u32(__float_as_uint(mx) & 0x7FFFFFFFu);
  if (lane == 0) sm.mx[warp] = wm;
  if (NEED_SUMS) {
    const float r = warp_sums4(pr, lane);
    const int j = (((lane & 1) * 2) + ((lane >> 1) & 1)) * 8 + warp;
    if (lane < 4) sm.s1[j] = r;
    else if (lane < 8) sm.s2[j] = r;
  }
  // the peers run before anything is written to their shared memory
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  __syncthreads();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 0) {
    const uint32_t m = warp_max_u32(sm.mx[lane & 7]);
    const float r1 = NEED_SUMS ? warp_tree_sum(sm.s1[lane]) : 0.f, r2 = NEED_SUMS ? warp_tree_sum(sm.s2[lane]) : 0.f;
    if (lane < ctas) {
      ClusterSmem* peer = cluster.map_shared_rank(&sm, lane);
      peer->pmx[rank] = m;
      peer->p1[rank] = r1;
      peer->p2[rank] = r2;
    }
  }
  cluster.sync();
  if (tid == 0) {
    uint32_t m = 0;
    for (int c = 0; c < ctas; ++c) m = max(m, sm.pmx[c]);
    const float S1 = NEED_SUMS ? smem_tree_sum(sm.p1, ctas) : 0.f, S2 = NEED_SUMS ? smem_tree_sum(sm.p2, ctas) : 0.f;
    const Scale sc = make_scale(m, S1, S2, len, a.b, a.clip_mode, a.clip_value);
    sm.sc.delta = sc.delta; sm.sc.rdelta = sc.rdelta; sm.sc.T = sc.T; sm.sc.lower = sc.lower;
    sm.sc.flags = sc.flags | (sc.T >= __uint_as_float(m) ? SCALE_NONE_OUTSIDE : 0u);
    if (rank == 0) {
      a.delta_out[worker] = sc.delta;
      if (sc.flags & 2u) atomicOr(a.dev_status, DEV_NONFINITE);
    }
  }
  __syncthreads();
  const ScaleRec sc = sm.sc;
  const bool degenerate = (sc.flags & 1u) != 0, count = !(sc.flags & SCALE_NONE_OUTSIDE) && a.count_clipped;
  const int words = (int)s.pad_words;
  uint32_t* out = a.codes + (int64_t)worker * a.stride_words;
  float fclip = 0.f;
#pragma unroll 1
  for (int it = 0; it < QITER; ++it) {
    if (rank * TILE + it * QGROUP >= len + 127) break;  // nothing of this sweep exists, padding words included
    const int j = j0 + it * QGROUP, g = j >> 3, nvalid = max(0, min(8, len - j));
    uint64_t lo = 0;
    if (!degenerate) {
      float sv[8];
      f32x2 w[4];
#pragma unroll
      for (int h = 0; h < 4; ++h) {  // v[it] without indexing registers by a variable
        w[h] = it == 0 ? v[0][h] : it == 1 ? v[1][h] : it == 2 ? v[2][h] : v[3][h];
      }
      if (count) scale_group8<true>(w, sc.rdelta, sc.T, sc.lower, fclip, sv);  // zero padding is inside the hull
      else scale_group8<false>(w, sc.rdelta, sc.T, sc.lower, fclip, sv);
      const U4 r = stream_block(a.seed, TAG_ROUND, (uint32_t)worker, a.k, s.block_base + (uint32_t)g);
      lo = quantize_scaled8<BITS>(sv, r);
      if (nvalid < 8) lo &= (1ull << (nvalid * BITS)) - 1ull;
    } else if (BITS > 1) {
      uint64_t zero = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) zero |= (1ull << (BITS - 1)) << (e * BITS);
      lo = nvalid < 8 ? zero & ((1ull << (nvalid * BITS)) - 1ull) : zero;
    }
    store_group_bounded<BITS>(out, g, lane, lo, words);
  }
  const uint32_t nclip = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)fclip);
  if (lane == 0) sm.clip[warp] = nclip;
  __syncthreads();
  if (tid == 0) {
    uint32_t n = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) n += sm.clip[w];
    cluster.map_shared_rank(&sm, 0)->pclip[rank] = n;
  }
  cluster.sync();
  if (rank == 0 && tid == 0) {
    uint32_t n = 0;
    for (int c = 0; c < ctas; ++c) n += sm.pclip[c];
    a.clipped_out[worker] = n;
  }
}

// b = 32: the message is the vector itself (clamped to [-T, T] when a clip rule is set).
__device__ __forceinline__ void bypass_tile(const QuantArgs& a, int tile, int worker, const ScaleRec& sc) {
  const int seg = a.tile_seg ? a.tile_seg[tile] : 0;
  const SegInfo s = a.segs[seg];
  const int64_t tstart = (int64_t)(tile - s.tile_first) * TILE;
  const float* p = a.U + (int64_t)worker * a.ld + s.off;
  const float* q = a.U_sub ? a.U_sub + (int64_t)worker * a.ld + s.off : nullptr;
  const bool vec = aligned16(p) && (!q || aligned16(q));
  const int tid = threadIdx.x, lane = tid & 31;
  uint32_t* out = a.codes + (int64_t)worker * a.stride_words + s.word_off;
  uint32_t nclip = 0;
  if (vec && tstart + TILE <= s.len) {  // four values per thread and access: neighbouring lanes fill whole lines
    const float *pt = p + tstart + tid * 4, *qt = q ? q + tstart + tid * 4 : nullptr;
    float4 v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __ldcs(reinterpret_cast<const float4*>(pt + i * QT * 4));
    if (qt) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 w = __ldcs(reinterpret_cast<const float4*>(qt + i * QT * 4));
        v[i] = make_float4(__fsub_rn(v[i].x, w.x), __fsub_rn(v[i].y, w.y), __fsub_rn(v[i].z, w.z), __fsub_rn(v[i].w, w.w));
      }
    }
    auto clamp = [&](float& x) {
      if (x > sc.T) { x = sc.T; ++nclip; }
      if (x < -sc.T) { x = -sc.T; ++nclip; }
    };
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (a.clip_mode != CLIP_NONE) { clamp(v[i].x); clamp(v[i].y); clamp(v[i].z); clamp(v[i].w); }
      *reinterpret_cast<float4*>(out + tstart + tid * 4 + i * QT * 4) = v[i];
    }
    if (a.clip_mode != CLIP_NONE) add_count(nclip, &a.clipped_out[(int64_t)worker * a.nseg + seg]);
    return;
  }
  float u[QITER][8];  // all loads before the first store
#pragma unroll
  for (int it = 0; it < QITER; ++it) load8(p, q, tstart + (int64_t)it * QGROUP + tid * 8, s.len, vec, u[it]);
#pragma unroll
  for (int it = 0; it < QITER; ++it) {
    const int64_t j = tstart + (int64_t)it * QGROUP + tid * 8;
    if (j >= s.pad_words) continue;
    float* v = u[it];
    if (a.clip_mode != CLIP_NONE) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (j + e < s.len) {
          if (v[e] > sc.T) { v[e] = sc.T; ++nclip; }
          if (v[e] < -sc.T) { v[e] = -sc.T; ++nclip; }
        }
      }
    }
    if (j + 8 <= s.len) {  // the stream starts on a 16-byte boundary
      *reinterpret_cast<float4*>(out + j) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<float4*>(out + j + 4) = make_float4(v[4], v[5], v[6], v[7]);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (j + e < s.pad_words) out[j + e] = (j + e < s.len) ? __float_as_uint(v[e]) : 0u;
    }
  }
  nclip = __reduce_add_sync(0xFFFFFFFFu, nclip);
  if (lane == 0 && nclip) atomicAdd(&a.clipped_out[(int64_t)worker * a.nseg + seg], nclip);
}

__global__ void __launch_bounds__(QT) bypass_kernel(QuantArgs a) {
  launch_dependents();
  wait_for_launch_before();
  const int tile = (int)(gridDim.x - 1 - blockIdx.x), worker = (int)(gridDim.y - 1 - blockIdx.y);  // from the end, as quantize_kernel
  const int seg = a.tile_seg ? a.tile_seg[tile] : 0;
  bypass_tile(a, tile, worker, a.scales[(int64_t)worker * a.nseg + seg]);
}

}  // namespace

// Where the first look's loads carry a cache policy, and how much is kept: three eighths of L2 of each input.  Quantizer, us, on the
// 126.5 MB of a B200, 8 workers, without / with 24, 36, 47 (three eighths), 60 and 100 MB kept: 134 MB of values, b = 4 54.6 / 51.7, 51.3,
// 51.8, 52.5, 54.6; 537 MB, b = 8 201.6 / 193.1, 192.8, 193.3, 193.5, 194.5.  With a subtrahend, without / with 48, 72, 95 and 120 MB:
// 537 MB, b = 4 168.1 / 166.3, 165.8, 165.2, 164.9.
// From: inputs beyond five eighths of L2 (each).  Shorter ones stay by themselves: 75 MB 34.5 / 34.7, 84 MB 38.0 / 37.8, 92 MB 41.5 / 40.4;
// with a subtrahend 134 MB together 47.0 / 47.0, 168 MB 57.4 / 56.8.
// To: what is saved does not grow with the input, while the loads cost a hundredth of the first look: 16 times L2 (2.0 GB 680.6 / 674.9,
// 2.1 GB 702.3 / 702.3), with a subtrahend 6 times (b = 4 / b = 8 without and with, 738 MB 226.2, 225.4 / 235.7, 234.1; 805 MB 246.3, 249.1 /
// 260.3, 258.9; 1.1 GB 326.2, 333.7 / 343.9, 345.6).
// Only where all rows and tensors start on 32-byte boundaries: the shorter loads of the others have no policy to carry (537 MB with
// every second row off 181.9 / 183.5).
int quantize_kept_tiles(const QuantArgs& a, bool offsets_aligned, int64_t l2_bytes) {
  auto aligned = [](const float* p) { return (reinterpret_cast<uintptr_t>(p) & 31u) == 0; };
  if (!offsets_aligned || !aligned(a.U) || !aligned(a.U_sub) || (a.N > 1 && a.ld % 8 != 0)) return 0;
  const int64_t tile_bytes = (int64_t)TILE * sizeof(float), bytes = (int64_t)a.N * a.ntiles * tile_bytes;  // of each input
  if (bytes <= l2_bytes / 8 * 5 || bytes * (a.U_sub ? 2 : 1) > l2_bytes * (a.U_sub ? 6 : 16)) return 0;
  return (int)(l2_bytes / 8 * 3 / tile_bytes);
}

// One cluster per worker: vectors of one segment and at most CTILES tiles, the fixed widths.  Up to about four CTAs per SM
// the clusters run side by side; with more of them the two passes over L2 of the other paths are as good.
bool quantize_fits_cluster(const QuantArgs& a, int sm_count) {
  const bool fixed_width = a.b == 1 || a.b == 2 || a.b == 3 || a.b == 4 || a.b == 8;
  return fixed_width && a.nseg == 1 && !a.shared_scale && a.ntiles >= 1 && a.ntiles <= CTILES && (int64_t)a.N * a.ntiles <= 4ll * sm_count;
}
cudaError_t launch_quantize_cluster(const QuantArgs& a, cudaStream_t st) {
  using ClusterKernel = void (*)(QuantArgs);
  const bool sums = a.clip_mode == CLIP_STD;
  ClusterKernel k;
  switch (a.b) {
    case 1: k = sums ? quantize_cluster_kernel<1, true> : quantize_cluster_kernel<1, false>; break;
    case 2: k = sums ? quantize_cluster_kernel<2, true> : quantize_cluster_kernel<2, false>; break;
    case 3: k = sums ? quantize_cluster_kernel<3, true> : quantize_cluster_kernel<3, false>; break;
    case 4: k = sums ? quantize_cluster_kernel<4, true> : quantize_cluster_kernel<4, false>; break;
    default: k = sums ? quantize_cluster_kernel<8, true> : quantize_cluster_kernel<8, false>; break;
  }
  int ctas = 1;
  while (ctas < a.ntiles) ctas <<= 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)ctas, (unsigned)a.N);
  cfg.blockDim = dim3(QT);
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)ctas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, k, a);
}

int quantize_run_tiles() { return QRUN; }

int quantize_pack_launches(const QuantArgs& a) {
  if (a.N <= 0 || a.nseg <= 0) return 0;
  return (a.ntiles > 0 ? 3 : 1) + (a.shared_scale ? 1 : 0);  // statistics, scale, codes; nothing but the scale of an empty vector
}

cudaError_t launch_quantize_pack(const QuantArgs& a, int kept_tiles, int sm_count, cudaStream_t st, LaunchHook hook, void* user) {
  if (a.N <= 0 || a.nseg <= 0) return cudaSuccess;
  const dim3 grid((unsigned)(a.ntiles > 0 ? a.ntiles : 1), (unsigned)a.N), block(QT);
  auto launch = [&](auto kernel, dim3 g, auto... args) { return launch_overlapped(kernel, g, block, 0, st, a, args...); };
  cudaError_t e = cudaSuccess;
  if (a.ntiles > 0) {
    if (hook) hook(user, 3 /* LPC_KERNEL_QUANT_STATS */, 1);
    const bool sums = a.clip_mode == CLIP_STD;
    if (kept_tiles > 0) e = sums ? launch(stats_kernel<true, true>, grid, kept_tiles) : launch(stats_kernel<false, true>, grid, kept_tiles);
    else e = sums ? launch(stats_kernel<true, false>, grid, 0) : launch(stats_kernel<false, false>, grid, 0);
    if (hook) hook(user, 3, 0);
    if (e != cudaSuccess) return e;
  }
  if (hook) hook(user, 5 /* LPC_KERNEL_OTHER */, 1);
  e = launch(finish_kernel, dim3((unsigned)a.nseg, (unsigned)a.N));
  if (hook) hook(user, 5, 0);
  if (e != cudaSuccess) return e;
  if (a.shared_scale) {
    if ((e = launch_overlapped(share_scale_kernel, dim3((unsigned)a.nseg), dim3(32), 0, st, a)) != cudaSuccess) return e;
  }
  if (a.ntiles <= 0) return cudaSuccess;
  struct Close {  // closes the timing scope of the second pass on every return path
    LaunchHook h; void* u;
    ~Close() { if (h) h(u, 4, 0); }
  } close_{hook, user};
  if (hook) hook(user, 4 /* LPC_KERNEL_QUANT_PACK */, 1);
  // Tiles per CTA: long runs read ahead better, but the last wave of CTAs (four to an SM) should be a small part of all:
  // as long as there are three waves (8 x 2^23: 103 us with two tiles, 119 with one; 8 x 2^24: 187 us with four, 195 with two).
  int run = QRUN;
  while (run > 1 && (int64_t)a.ntiles * a.N < 3ll * run * 4 * sm_count) run >>= 1;
  const dim3 runs((unsigned)((a.ntiles + run - 1) / run), (unsigned)a.N);
  auto pack = [&](auto width) {
    constexpr int B = decltype(width)::value;
    return a.count_clipped ? launch(quantize_kernel<B, true>, runs, run) : launch(quantize_kernel<B, false>, runs, run);
  };
  switch (a.b) {
    case 1: return pack(std::integral_constant<int, 1>());
    case 2: return pack(std::integral_constant<int, 2>());
    case 3: return pack(std::integral_constant<int, 3>());
    case 4: return pack(std::integral_constant<int, 4>());
    case 8: return pack(std::integral_constant<int, 8>());
    case 32: return launch(bypass_kernel, grid);
    default: return pack(std::integral_constant<int, 0>());
  }
}

}  // namespace lpc

namespace lpc {
namespace {
__global__ void stream_blocks_kernel(uint64_t seed, uint32_t tag, uint32_t worker, uint64_t k, uint32_t block0,
                                     int64_t count, uint32_t* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) {
    const U4 r = stream_block(seed, tag, worker, k, block0 + (uint32_t)i);
    out[4 * i + 0] = r.x; out[4 * i + 1] = r.y; out[4 * i + 2] = r.z; out[4 * i + 3] = r.w;
  }
}

__global__ void loop_scales_kernel(const uint32_t* __restrict__ max_bits, const float* __restrict__ S1, const float* __restrict__ S2,
                                   int64_t count, ScaleRule rule, int b, int clip_mode, float clip_value,
                                   float4* __restrict__ scale_out, uint32_t* __restrict__ flags_out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const uint32_t m = max_bits[i];
  const Scale sc = make_scale_in_loop(m, S1[i], S2[i], rule, b, clip_mode, clip_value);
  float T;
  const bool doubles = clip_mode == CLIP_STD && m != 0u && m < 0x7F800000u &&
                       !std_threshold_single(S1[i], S2[i], rule, clip_value, __uint_as_float(m), T);
  scale_out[i] = make_float4(sc.delta, sc.rdelta, sc.T, sc.lower);
  flags_out[i] = sc.flags | (doubles ? 4u : 0u);
}
}  // namespace

cudaError_t launch_loop_scales(const uint32_t* max_bits, const float* S1, const float* S2, int64_t count, const ScaleRule& rule, int b,
                               int clip_mode, float clip_value, float4* scale_out, uint32_t* flags_out, cudaStream_t st) {
  loop_scales_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(max_bits, S1, S2, count, rule, b, clip_mode, clip_value, scale_out,
                                                                     flags_out);
  return cudaGetLastError();
}

cudaError_t launch_stream_blocks(uint64_t seed, uint32_t tag, uint32_t worker, uint64_t k, uint32_t block0,
                                 int64_t count, uint32_t* out, cudaStream_t st) {
  stream_blocks_kernel<<<(unsigned)((count + 255) / 256), 256, 0, st>>>(seed, tag, worker, k, block0, count, out);
  return cudaGetLastError();
}
}  // namespace lpc
