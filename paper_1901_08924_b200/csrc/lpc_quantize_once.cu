// Quantization step of Algorithm 1 (step 7) of u = U - U_sub with ONE look at the values, for many messages (tensors of many workers) that
// together are longer than L2: u waits in shared memory from the statistics to the codes, so that both inputs are read once.
//
// One CTA per SM takes every gridDim-th tile.  A tile comes by a bulk copy into one of seven slots of a whole tile each, and leaves it with
// its codes.  22 warps take units of 512 values: the difference and its statistics as soon as the tile is there, the codes three rounds
// (about four tiles) later.  All CTAs walk through the messages in the same order, so a message's tiles are looked at everywhere within a
// few turns, and its scale is known when its codes are due.  Six more warps with one task each keep the hand-overs out of the others' way:
// copies (and prefetches to L2), tile partials to the other CTAs, scales (three warps), counts and slots given back.
//
// Tile partials are 16-byte words with a tag that names the call, so nothing is cleared and nothing is fenced.  No CTA relies on another one
// running: whoever waits too long for a tile's partials forms them from memory by itself.
//
// What bounds it: how long a tile stays in its slot (load 1.2 us, statistics until its partials are out 3, until its scale is there 5, codes
// 1.5) times one tile per 2.0 us and SM, where the copy rate would allow one per 1.5.  62 tensors of an 18-layer residual network, 16 workers,
// b = 4: 328 us against 450 for two looks in three launches.  Tried: 16 warps a tile at a time 351 (all in the same phase, idle pipes), two
// teams of eight 387, 24 warps 417 (64 registers), 16 to 24 warps with a lag of two to five rounds 332 to 420, one CTA per message
// that forms its scale for all 616; looks at the partials before they can be there, 916, keep L2 busy; statistics and codes as CTAs of
// their own, the codes 900 tiles behind in L2, 537 (both keep their bytes in flight in registers).  Without a subtrahend the same kernel takes
// 264 against 260 us: there the two looks are half as many bytes.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "lpc_quantize.cuh"

namespace lpc {
namespace {

constexpr int SLOTS = 7;
constexpr int CW = 22;           // warps that form statistics and codes
constexpr int UNIT = 512;        // consecutive values that such a warp takes at a time, two groups of eight per lane
constexpr int UNITS = TILE / UNIT;
constexpr int LAG = 3;           // rounds of all these warps between a unit's statistics and its codes
constexpr int SCALERS = 3;
constexpr int W_COPY = CW, W_PUBLISH = CW + 1, W_SCALE = CW + 2, W_COUNT = W_SCALE + SCALERS;
constexpr int OT = (W_COUNT + 1) * 32;
constexpr int ROWS = 10;         // a message has at most 32 * ROWS tiles
constexpr uint64_t HELP_NS = 50000;  // a tile whose partials do not come for this long is looked at here

static_assert(32 * ROWS * TILE < 1 << 24, "lengths are exact in single precision");

struct TileInfo {
  const float* p;     // the tile's first value
  const float* q;     // of the subtrahend
  uint32_t* out;      // the tile's first word
  int valid, words;   // values of the tile, words from `out` on
  uint32_t block0;    // first Philox block
  int worker, msg;    // message: worker * nseg + segment
  int tiles;          // of the message
};

struct OnceSmem {
  uint64_t full[SLOTS];   // the tile's values have arrived
  uint64_t known[SLOTS];  // `info` of the slot's next tile is written
  uint64_t summed[SLOTS]; // all warps' partials of the tile are there
  uint64_t scaled[SLOTS]; // `scale` is written
  uint64_t coded[SLOTS];  // all warps have formed their codes
  uint64_t empty[SLOTS];  // the slot may be used again
  TileInfo info[SLOTS];
  ScaleRec scale[SLOTS];
  float s1[SLOTS][UNITS], s2[SLOTS][UNITS];
  uint32_t mx[SLOTS][UNITS];
  uint32_t clip[SLOTS];
  uint32_t tag;
  int failed;
};

// The caller's place in the sequence of tiles: worker by worker, a worker's tiles in order.
struct Walk {
  int worker, tile;
  __device__ __forceinline__ Walk(int first, int ntiles) : worker(first / ntiles), tile(first % ntiles) {}
  __device__ __forceinline__ void advance(int by, int ntiles) {
    tile += by;
    while (tile >= ntiles) {
      tile -= ntiles;
      ++worker;
    }
  }
};

// A tile's partials and the call's tag: one 16-byte word, written and read as a whole.
__device__ __forceinline__ void st_partials(ulonglong2* w, uint32_t mx, float s1, float s2, uint32_t tag) {
  const unsigned long long lo = (unsigned long long)__float_as_uint(s1) << 32 | mx, hi = (unsigned long long)tag << 32 | __float_as_uint(s2);
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(w), "l"(lo), "l"(hi) : "memory");
}
__device__ __forceinline__ void ld_partials(const ulonglong2* w, unsigned long long& lo, unsigned long long& hi) {
  asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}" : "=l"(lo), "=l"(hi) : "l"(w) : "memory");
}

// A tile's partials by one warp from memory; all lanes get them.
template <bool SUMS>
__device__ __noinline__ void tile_partials(const float* p, const float* q, int valid, uint32_t& mx_out, float& s1_out, float& s2_out) {
  const int lane = threadIdx.x & 31;
  float mx = 0.f, s1 = 0.f, s2 = 0.f;
#pragma unroll 1
  for (int i = 0; i < TILE / 256; ++i) {  // 256 values; lane i keeps their sums
    float u[8];
    load8(p, q, i * 256 + lane * 8, valid, true, u);
    const f32x2 v[4] = {pack2(u[0], u[1]), pack2(u[2], u[3]), pack2(u[4], u[5]), pack2(u[6], u[7])};
    float a, b;
    unpack2(stats_group8<SUMS>(v, mx), a, b);
    if constexpr (SUMS) {
      a = warp_tree_sum(a);
      b = warp_tree_sum(b);
      if (lane == i) { s1 = a; s2 = b; }
    }
  }
  mx_out = warp_max_u32(__float_as_uint(mx) & 0x7FFFFFFFu);
  s1_out = SUMS ? warp_tree_sum(s1) : 0.f;
  s2_out = SUMS ? warp_tree_sum(s2) : 0.f;
}

// Some CTA has not come as far as this tile, or has not even started: the tile is looked at here.
template <bool SUMS>
__device__ __noinline__ void help(const QuantOnceArgs& oa, int worker, const SegInfo& g, int tile, uint32_t tag) {
  const QuantArgs& a = oa.q;
  const int64_t off = (int64_t)worker * a.ld + g.off + (int64_t)tile * TILE;
  uint32_t mx;
  float s1, s2;
  tile_partials<SUMS>(a.U + off, a.U_sub + off, (int)min((int64_t)TILE, g.len - (int64_t)tile * TILE), mx, s1, s2);
  if ((threadIdx.x & 31) == 0) st_partials(oa.partials + (int64_t)worker * a.ntiles + g.tile_first + tile, mx, s1, s2, tag);
  __syncwarp();
}

// A group that reaches past the end of its tensor: straight from memory.
struct Group { f32x2 v[4]; };
__device__ __noinline__ Group ragged_group(const float* p, const float* q, int j, int valid) {
  float u[8];
  load8(p, q, j, valid, false, u);
  return Group{{pack2(u[0], u[1]), pack2(u[2], u[3]), pack2(u[4], u[5]), pack2(u[6], u[7])}};
}
__device__ __noinline__ ulonglong2 zero_group(int b, int valid) {  // a group of zero codes
  uint64_t lo = 0, hi = 0;
  for (int e = min(8, valid) - 1; e >= 0 && b > 1; --e) push_code(lo, hi, 1u << (b - 1), b);
  return make_ulonglong2(lo, hi);
}
__device__ __forceinline__ void give_up(volatile int* failed, unsigned int* dev_status) {
  atomicOr(dev_status, DEV_TIMEOUT);
  __threadfence();  // the CTA that ends the launch sees it: it counts this one among those that are through
  *failed = 1;
}
// Out of line, so that the code that every warp walks through stays small.  False: this wait or another one of the CTA ran out (the status
// word says so).  Whoever gets that goes no further: what it waited for, pointers among it, may never have been written.
__device__ __noinline__ bool slow_wait(uint64_t* bar, uint32_t parity, volatile int* failed, unsigned int* dev_status) {
  for (int i = 0; i < 200; ++i) {  // two seconds; the CTA's other waits end within a hundredth of one
    if (*failed) return false;
    if (mbar_wait(bar, parity, 10000000ull)) return true;
  }
  give_up(failed, dev_status);
  return false;
}

__device__ __forceinline__ void lds_pairs(const float* s, f32x2& a, f32x2& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(smem_u32(s)) : "memory");
}
__device__ __forceinline__ void sts_pairs(float* s, f32x2 a, f32x2 b) {
  asm volatile("st.shared.v2.b64 [%0], {%1, %2};" ::"r"(smem_u32(s)), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void ldg_pairs(const float* p, f32x2& a, f32x2& b) {
  asm volatile("ld.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
}

template <int BITS, bool SUMS>
__global__ void __launch_bounds__(OT, 1) quantize_once_kernel(QuantOnceArgs oa) {
  const QuantArgs& a = oa.q;
  extern __shared__ __align__(128) unsigned char once_smem[];
  float* slots = reinterpret_cast<float*>(once_smem);
  OnceSmem& sm = *reinterpret_cast<OnceSmem*>(once_smem + (size_t)SLOTS * TILE * 4);
  launch_dependents();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = (int)gridDim.x, total = a.N * a.ntiles;
  const int n = (total - (int)blockIdx.x + G - 1) / G;  // tiles of this CTA
  if (tid < SLOTS) {
    mbar_init(&sm.full[tid], 1);
    mbar_init(&sm.known[tid], 1);
    mbar_init(&sm.summed[tid], UNITS);
    mbar_init(&sm.scaled[tid], 1);
    mbar_init(&sm.coded[tid], UNITS);
    mbar_init(&sm.empty[tid], 2);  // the counts are taken and the partials are read
    mbar_fence_init();
    sm.clip[tid] = 0u;
  }
  wait_for_launch_before();
  if (tid == 0) {
    sm.failed = 0;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(sm.tag) : "l"(oa.epoch) : "memory");
  }
  __syncthreads();
  const uint32_t tag = sm.tag;
  auto lane_waits = [&](uint64_t* bar, uint32_t parity) {  // one thread
    return mbar_test(bar, parity) || slow_wait(bar, parity, &sm.failed, a.dev_status);
  };
  auto warp_waits = [&](uint64_t* bar, uint32_t parity) {  // a whole warp, which goes on together or not at all
    if (__all_sync(0xFFFFFFFFu, mbar_test(bar, parity))) return true;
    return (bool)__all_sync(0xFFFFFFFFu, slow_wait(bar, parity, &sm.failed, a.dev_status));
  };
  auto parity_of = [](int i) { return (uint32_t)((i / SLOTS) & 1); };

  if (warp < CW) {
    // ---- statistics of one unit, then codes of the one LAG rounds before.  Warp w takes the units w, w + CW, ... of the CTA's tiles; the
    // warps are at different places, so that the long chains of the statistics and the busy pipes of the codes overlap.
    struct Place {
      int i, part, s;    // tile, unit of it, its slot
      uint32_t parity;
      __device__ __forceinline__ void advance() {
        constexpr int STEP = CW / UNITS, REST = CW % UNITS;
        static_assert(STEP + 1 < SLOTS, "one wrap at most");
        part += REST;
        int by = STEP;
        if (part >= UNITS) { part -= UNITS; ++by; }
        i += by;
        s += by;
        if (s >= SLOTS) { s -= SLOTS; parity ^= 1u; }
      }
    };
    const int first = (lane & 4) ? 4 : 0;  // half of a group read first, so that a quarter warp's loads touch all banks
    auto statistics = [&](const Place& at) {
      const int s = at.s, own = at.part * UNIT + lane * 8;  // this thread's groups: `own` and own + 256
      float* slot = slots + (size_t)s * TILE;
      if (!warp_waits(&sm.known[s], at.parity)) return false;
      const int valid = sm.info[s].valid;
      f32x2 qv[2][4];
      const float* q = sm.info[s].q;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = own + h * 256;
        if (j + 8 <= valid) {
          ldg_pairs(q + j + first, qv[h][0], qv[h][1]);
          ldg_pairs(q + j + (4 - first), qv[h][2], qv[h][3]);
        }
      }
      if (!warp_waits(&sm.full[s], at.parity)) return false;
      float mx = 0.f;
      f32x2 pr[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int j = own + h * 256;
        f32x2 v[4];
        if (j + 8 <= valid) {
          lds_pairs(slot + j + first, v[0], v[1]);
          lds_pairs(slot + j + (4 - first), v[2], v[3]);
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = sub2_rn(v[e], qv[h][e]);
          sts_pairs(slot + j + first, v[0], v[1]);
          sts_pairs(slot + j + (4 - first), v[2], v[3]);
        } else {
          const Group g = ragged_group(sm.info[s].p, sm.info[s].q, j, valid);
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = g.v[e];
        }
        pr[h] = stats_group8<SUMS>(v, mx);  // exchanged halves only swap the operands of the tree's last addition
      }
      const uint32_t m = warp_max_u32(__float_as_uint(mx) & 0x7FFFFFFFu);
      if constexpr (SUMS) {
        const bool u0 = lane & 1, u1 = lane & 2;
        const f32x2 k = add2_rn(u0 ? pr[1] : pr[0], __shfl_xor_sync(0xFFFFFFFFu, u0 ? pr[0] : pr[1], 1));
        float x, y;
        unpack2(k, x, y);
        float r = add_rn(u1 ? y : x, __shfl_xor_sync(0xFFFFFFFFu, u1 ? x : y, 2));
        r = add_rn(r, __shfl_xor_sync(0xFFFFFFFFu, r, 4));
        r = add_rn(r, __shfl_xor_sync(0xFFFFFFFFu, r, 8));
        r = add_rn(r, __shfl_xor_sync(0xFFFFFFFFu, r, 16));
        r = add_rn(r, __shfl_xor_sync(0xFFFFFFFFu, r, 1));
        if (lane == 0) sm.s1[s][at.part] = r;
        if (lane == 2) sm.s2[s][at.part] = r;
      }
      if (lane == 0) sm.mx[s][at.part] = m;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.summed[s]);
      return true;
    };
    auto codes = [&](const Place& at) {
      const int s = at.s, own = at.part * UNIT + lane * 8;
      float* slot = slots + (size_t)s * TILE;
      if (!warp_waits(&sm.scaled[s], at.parity)) return false;
      const TileInfo& t = sm.info[s];
      const ScaleRec sc = sm.scale[s];
      const int valid = t.valid, words = t.words, b = BITS ? BITS : a.b;
      uint32_t* out = t.out;
      float fclip = 0.f;
      uint64_t lo[2] = {0, 0}, hi[2] = {0, 0};
      if (sc.flags & 1u) {  // degenerate: zero codes
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const ulonglong2 z = zero_group(b, valid - own - h * 256);
          lo[h] = z.x;
          hi[h] = z.y;
        }
      } else {
        f32x2 v[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int j = own + h * 256;
          if (j + 8 <= valid) {
            lds_pairs(slot + j, v[h][0], v[h][1]);
            lds_pairs(slot + j + 4, v[h][2], v[h][3]);
          } else {
            const Group g = ragged_group(t.p, t.q, j, valid);
#pragma unroll
            for (int e = 0; e < 4; ++e) v[h][e] = g.v[e];
          }
        }
        U4 r[2];
        float sv[2][8];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          r[h] = stream_block(a.seed, TAG_ROUND, (uint32_t)t.worker, a.k, t.block0 + (uint32_t)((own >> 3) + h * 32));
        if ((sc.flags & SCALE_NONE_OUTSIDE) || !a.count_clipped) {
#pragma unroll
          for (int h = 0; h < 2; ++h) scale_group8<false>(v[h], sc.rdelta, sc.T, sc.lower, fclip, sv[h]);
        } else {
#pragma unroll
          for (int h = 0; h < 2; ++h) scale_group8<true>(v[h], sc.rdelta, sc.T, sc.lower, fclip, sv[h]);  // zeros past the end are inside the hull
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if constexpr (BITS != 0) lo[h] = quantize_scaled8<BITS ? BITS : 1>(sv[h], r[h]);
          else quantize_scaled8_rt(sv[h], r[h], b, lo[h], hi[h]);
        }
        if (valid < TILE) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int bits = max(0, min(8, valid - (own + h * 256))) * b;  // nothing but zeros past the end
            if (bits < 64) { lo[h] &= (1ull << bits) - 1ull; hi[h] = 0; }
            else if (bits < 128) hi[h] &= (1ull << (bits - 64)) - 1ull;
          }
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if constexpr (BITS != 0) {
          const int g = (own >> 3) + h * 32;
          store_group_bounded<BITS ? BITS : 1>(out, g, lane, lo[h], words);
        } else {  // these values have been read: their place in the slot puts the words together
          const int w0 = (at.part * 16 + h * 8) * b;
          store_any_width(out + w0, words - w0, lo[h], hi[h], b, lane, lane, reinterpret_cast<uint8_t*>(slot + at.part * UNIT));
        }
      }
      const uint32_t nclip = __reduce_add_sync(0xFFFFFFFFu, (uint32_t)fclip);
      fence_proxy_async();  // the slot was written by this thread; a bulk copy is next
      __syncwarp();
      if (lane == 0) {
        if (nclip) atomicAdd(&sm.clip[s], nclip);
        mbar_arrive(&sm.coded[s]);
      }
      return true;
    };
    Place now = {warp / UNITS, warp % UNITS, warp / UNITS, 0u}, then = now;
    int behind = LAG;
#pragma unroll 1
    while (then.i < n) {
      if (now.i < n) {
        if (!statistics(now)) break;
        now.advance();
      }
      if (behind > 0) {
        --behind;
      } else {
        if (!codes(then)) break;
        then.advance();
      }
    }
  } else if (warp == W_COPY) {
    // ---- copies: a slot is filled again as soon as it has been given back; the tile after it is on its way to L2 by then ------
    if (lane == 0) {
      Walk w(blockIdx.x, a.ntiles);
      auto describe = [&] {
        const int seg = a.tile_seg ? a.tile_seg[w.tile] : 0;
        const SegInfo g = a.segs[seg];
        const int64_t t0 = (int64_t)(w.tile - g.tile_first) * TILE, word0 = (t0 >> 5) * (BITS ? BITS : a.b);
        TileInfo t;
        t.p = a.U + (int64_t)w.worker * a.ld + g.off + t0;
        t.q = a.U_sub + (int64_t)w.worker * a.ld + g.off + t0;
        t.out = a.codes + (int64_t)w.worker * a.stride_words + g.word_off + word0;
        t.valid = (int)min((int64_t)TILE, g.len - t0);
        t.words = (int)min((int64_t)TILE, g.pad_words - word0);
        t.block0 = g.block_base + (uint32_t)(t0 >> 3);
        t.worker = w.worker;
        t.msg = w.worker * a.nseg + seg;
        t.tiles = g.tile_count;
        const uint32_t bytes = (uint32_t)(t.valid & ~3) * 4u;
        if (bytes) {
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(t.p), "r"(bytes) : "memory");
          asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(t.q), "r"(bytes) : "memory");
        }
        return t;
      };
      TileInfo next = describe();
      int issued = 0;
#pragma unroll 1
      for (int i = 0; i < n; ++i) {
        const int s = i % SLOTS;
        const TileInfo t = next;
        if (i + 1 < n) {
          w.advance(G, a.ntiles);
          next = describe();
        }
        if (i == oa.stop_at && blockIdx.x == 0) {  // inspection of what follows a wait that ran out
          give_up(&sm.failed, a.dev_status);
          break;
        }
        if (i >= SLOTS && !lane_waits(&sm.empty[s], parity_of(i - SLOTS))) break;
        sm.info[s] = t;
        mbar_arrive(&sm.known[s]);
        const uint32_t bytes = (uint32_t)(t.valid & ~3) * 4u;  // a ragged end of less than 16 bytes is read by whoever needs it
        mbar_expect_tx(&sm.full[s], bytes);
        if (bytes) bulk_load(slots + (size_t)s * TILE, t.p, bytes, &sm.full[s]);
        issued = i + 1;
      }
      // no CTA leaves with copies on their way: they have all landed where nothing failed, and get a bounded chance where something did
      for (int i = max(0, issued - SLOTS); i < issued; ++i) mbar_wait(&sm.full[i % SLOTS], parity_of(i), 100000000ull);
    }
  } else if (warp == W_PUBLISH) {
    // ---- a tile's partials to whoever needs them ---------------------------------------------------------------------
    if (blockIdx.x == 0) {  // tensors without a single value
      for (int m = lane; m < a.N * a.nseg; m += 32) {
        if (a.segs[m % a.nseg].tile_count == 0) {
          a.delta_out[m] = 0.f;
          a.clipped_out[m] = 0u;
        }
      }
    }
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const int s = i % SLOTS;
      if (!warp_waits(&sm.summed[s], parity_of(i))) break;
      float s1 = SUMS ? sm.s1[s][lane & (UNITS - 1)] : 0.f, s2 = SUMS ? sm.s2[s][lane & (UNITS - 1)] : 0.f;
      const uint32_t m = warp_max_u32(sm.mx[s][lane & (UNITS - 1)]);
      if constexpr (SUMS) {
#pragma unroll
        for (int x = 1; x < UNITS; x <<= 1) {
          s1 = add_rn(s1, __shfl_xor_sync(0xFFFFFFFFu, s1, x));
          s2 = add_rn(s2, __shfl_xor_sync(0xFFFFFFFFu, s2, x));
        }
      }
      if (lane == 0) {
        st_partials(oa.partials + (int64_t)blockIdx.x + (int64_t)i * G, m, s1, s2, tag);
        mbar_arrive(&sm.empty[s]);
      }
    }
  } else if (warp < W_COUNT) {
    // ---- scales: warp c of these takes the tiles c, c + SCALERS, ... -------------------------------------------------
    const int c = warp - W_SCALE;
    Walk w((int)blockIdx.x, a.ntiles);
    w.advance(c * G, a.ntiles);
    int last = -1;
    ScaleRec rec = {};
#pragma unroll 1
    for (int i = c; i < n; i += SCALERS, w.advance(SCALERS * G, a.ntiles)) {
      const int s = i % SLOTS;
      const int seg = a.tile_seg ? a.tile_seg[w.tile] : 0, msg = w.worker * a.nseg + seg;
      if (msg != last) {
        const SegInfo g = a.segs[seg];
        const int count = g.tile_count;
        const ulonglong2* from = oa.partials + (int64_t)w.worker * a.ntiles + g.tile_first;
        // Nobody looks at other CTAs' partials before this CTA's are out, nor at all of them before the last tile's are there: looks that
        // come too early keep L2 busy.
        if (!warp_waits(&sm.summed[s], parity_of(i))) break;
        {
          uint64_t since = 0;
#pragma unroll 1
          for (uint32_t it = 0;; ++it) {
            unsigned long long lo, hi;
            ld_partials(from + count - 1, lo, hi);
            if ((uint32_t)(hi >> 32) == tag) break;
            if ((it & 63u) == 63u) {
              const uint64_t now = global_ns();
              if (since == 0) since = now;
              if (now - since >= HELP_NS) break;
            }
            __nanosleep(64);
          }
          __syncwarp();
        }
        // lane l takes the tiles 32 k + l, all of them in flight together
        unsigned long long lo[ROWS], hi[ROWS];
        uint64_t since = 0;
#pragma unroll 1
        for (uint32_t it = 0;; ++it) {
          bool ok = true;
#pragma unroll
          for (int k = 0; k < ROWS; ++k) {
            lo[k] = 0;
            hi[k] = (unsigned long long)tag << 32;
            if (k * 32 + lane < count) ld_partials(from + k * 32 + lane, lo[k], hi[k]);
          }
#pragma unroll
          for (int k = 0; k < ROWS; ++k) ok = ok && (uint32_t)(hi[k] >> 32) == tag;
          if (__all_sync(0xFFFFFFFFu, ok)) break;
          if ((it & 63u) != 63u) continue;
          const uint64_t now = __shfl_sync(0xFFFFFFFFu, global_ns(), 0);
          if (since == 0) since = now;
          if (now - since < HELP_NS) continue;
          int missing = 0;
#pragma unroll
          for (int k = ROWS - 1; k >= 0; --k)
            if ((uint32_t)(hi[k] >> 32) != tag) missing = k * 32 + lane;
          const int who = __ffs(__ballot_sync(0xFFFFFFFFu, !ok)) - 1;
          help<SUMS>(oa, w.worker, g, __shfl_sync(0xFFFFFFFFu, missing, who), tag);
        }
        uint32_t mx = 0;
        float S1 = 0.f, S2 = 0.f;
#pragma unroll
        for (int k = 0; k < ROWS; ++k) mx = max(mx, (uint32_t)lo[k]);
        mx = warp_max_u32(mx);
        if constexpr (SUMS) {  // the tree over the lanes of each row, then over the rows
          auto sums = [&](auto rows) {
            constexpr int V = decltype(rows)::value;
            float x[V], y[V];
#pragma unroll
            for (int k = 0; k < V; ++k) {
              x[k] = k < ROWS ? __uint_as_float((uint32_t)(lo[k < ROWS ? k : 0] >> 32)) : 0.f;
              y[k] = k < ROWS ? __uint_as_float((uint32_t)hi[k < ROWS ? k : 0]) : 0.f;
            }
            WarpHalving<V, 0>::run(x, lane);
            WarpHalving<V, 0>::run(y, lane);
            S1 = x[0];
            S2 = y[0];
#pragma unroll
            for (int m = V / 2; m >= 1; m >>= 1) {
              S1 = add_rn(S1, __shfl_xor_sync(0xFFFFFFFFu, S1, m));
              S2 = add_rn(S2, __shfl_xor_sync(0xFFFFFFFFu, S2, m));
            }
          };
          if (count <= 128) sums(std::integral_constant<int, 4>());
          else sums(std::integral_constant<int, 16>());
        }
        const float flen = (float)g.len, inv = __frcp_rn(flen);  // exact: a message here has fewer than 2^24 values
        const ScaleRule rule = {g.len, inv, mul_rn(__fmaf_rn(-inv, flen, 1.f), inv), oa.levels, oa.inv_levels};
        const Scale sc = make_scale_in_loop(mx, S1, S2, rule, a.b, a.clip_mode, a.clip_value);
        rec.delta = sc.delta; rec.rdelta = sc.rdelta; rec.T = sc.T; rec.lower = sc.lower;
        rec.flags = sc.flags | (sc.T >= __uint_as_float(mx) ? SCALE_NONE_OUTSIDE : 0u);
        last = msg;
        if (w.tile == g.tile_first && lane == 0) {
          a.delta_out[msg] = sc.delta;
          if (sc.flags & 2u) atomicOr(a.dev_status, DEV_NONFINITE);
        }
      }
      if (!warp_waits(&sm.known[s], parity_of(i))) break;  // the slot is this tile's: nobody reads the scale of the one before any more
      if (lane == 0) {
        sm.scale[s] = rec;
        mbar_arrive(&sm.scaled[s]);
      }
      __syncwarp();
    }
  } else if (lane == 0) {
    // ---- counts of coordinates outside the hull, and slots given back.  A message's counter holds the count and, above it, the
    // tiles that have been added; whoever adds the last one writes the result and clears the counter for the next call.
    int msg = -1, tiles = 0, of = 0;
    uint32_t cnt = 0;
    auto flush = [&] {
      if (msg < 0 || !a.count_clipped) return;
      const unsigned long long mine = ((unsigned long long)tiles << 40) | cnt;
      const unsigned long long sum = atomicAdd(oa.counts + msg, mine) + mine;
      if ((int)(sum >> 40) == of) {
        a.clipped_out[msg] = (uint32_t)sum;
        oa.counts[msg] = 0ull;
      }
    };
#pragma unroll 1
    for (int i = 0; i < n; ++i) {
      const int s = i % SLOTS;
      if (!lane_waits(&sm.coded[s], parity_of(i))) break;
      const int m = sm.info[s].msg, t = sm.info[s].tiles;
      const uint32_t c = sm.clip[s];
      sm.clip[s] = 0u;
      mbar_arrive(&sm.empty[s]);
      if (m != msg) {
        flush();
        msg = m; of = t; tiles = 0; cnt = 0;
      }
      tiles += 1;
      cnt += c;
    }
    flush();
    // the last CTA of the grid moves the tag on
    __threadfence();
    if (atomicInc(oa.done, (unsigned)G - 1u) == (unsigned)G - 1u) {
      __threadfence();
      // where a wait ran out tiles are missing from some messages' counters, which the next call would go on from
      if (*(volatile unsigned int*)a.dev_status & DEV_TIMEOUT)
        for (int m = 0; m < a.N * a.nseg; ++m) oa.counts[m] = 0ull;
      *oa.epoch = tag == 0xFFFFFFFFu ? 1u : tag + 1u;
    }
  }
}

template <int BITS, bool SUMS>
cudaError_t launch_t(const QuantOnceArgs& oa, int grid, cudaStream_t st) {
  constexpr size_t smem = (size_t)SLOTS * TILE * 4 + sizeof(OnceSmem);
  static_assert(smem <= 227 * 1024, "shared memory of one CTA");
  static std::atomic<bool> allowed[64];  // the attribute is raised once per device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64 || !allowed[dev].load(std::memory_order_relaxed)) {
    e = cudaFuncSetAttribute(quantize_once_kernel<BITS, SUMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    if (dev >= 0 && dev < 64) allowed[dev].store(true, std::memory_order_relaxed);
  }
  return launch_overlapped(quantize_once_kernel<BITS, SUMS>, dim3((unsigned)grid), dim3(OT), smem, st, oa);
}

}  // namespace

// From: inputs beyond three quarters of L2 each (three launches / one, us, 16 workers, b = 4, each input 64 MB 41.0 / 43.5, 76 MB 48.5 / 47.8,
// 84 MB 53.1 / 52.5, 96 MB 58.7 / 56.7, 120 MB 74.1 / 68.1, 200 MB 115 / 89): shorter ones find part of the second look in L2.
// Messages of at most two tiles per SM, so that their tiles are all looked at within the lag (120 MB in messages of 40 tiles 74.3 / 64.4, 148
// 70.4 / 64.4, 296 71.3 / 65.4).  Tiles full to seven eighths on average: a tile takes its turn however few values it has (300 tensors of
// 16,384 values 205 / 156, of 12,000 163 / 170, 1,500 of 2,000 255 / 563).
// Without 16-byte boundaries there are no bulk copies.
bool quantize_takes_one_look(const QuantArgs& a, int64_t len, int max_tiles, bool offsets_x4, int sm_count, int64_t l2_bytes) {
  auto aligned = [](const float* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  if (!a.U_sub || a.b == 32 || a.shared_scale || !offsets_x4 || !aligned(a.U) || !aligned(a.U_sub) || (a.N > 1 && a.ld % 4 != 0)) return false;
  return (int64_t)a.N * len * 4 > l2_bytes / 4 * 3 && max_tiles <= std::min(2 * sm_count, 32 * ROWS) && len * 8 >= (int64_t)a.ntiles * TILE * 7 &&
         (int64_t)a.N * a.ntiles <= 0x7FFFFFFF;
}

cudaError_t launch_quantize_once(const QuantOnceArgs& oa, int sm_count, cudaStream_t st) {
  const int grid = (int)std::min<int64_t>(sm_count, (int64_t)oa.q.N * oa.q.ntiles);
  auto run = [&](auto width) {
    constexpr int B = decltype(width)::value;
    return oa.q.clip_mode == CLIP_STD ? launch_t<B, true>(oa, grid, st) : launch_t<B, false>(oa, grid, st);
  };
  switch (oa.q.b) {
    case 1: return run(std::integral_constant<int, 1>());
    case 2: return run(std::integral_constant<int, 2>());
    case 3: return run(std::integral_constant<int, 3>());
    case 4: return run(std::integral_constant<int, 4>());
    case 8: return run(std::integral_constant<int, 8>());
    default: return run(std::integral_constant<int, 0>());
  }
}

}  // namespace lpc
