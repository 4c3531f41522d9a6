// The whole inner loop of Algorithm 1 or 2 in one launch for minibatches whose rows stream through shared memory: more than 64 rows per
// worker (up to 256), or fewer where the loop with resident rows has no room.  It joins the streaming worker kernel of lpc_inner.cu (warps
// specialised by role, a ring of stages, hand-overs as mbarrier phases) with the tagged words of lpc_persist.cu (codes, scales and the second
// estimator travel between the clusters through L2).
//
// The groups of rows of all steps form one stream: while a step ends (statistics, scale, codes, the other workers' words, the new point) the
// ring fills with the next step's rows, whose indices depend on the iteration number alone.  Single launches leave memory idle from the last
// row of a step until the next launch has started.
//
// A group is as many rows as make up a stage: 4 rows of a slice of 2,048 columns, 32 of one of 256 or 128, because a group costs its chain of
// hand-overs whatever its bytes.  Each warp issues a bulk copy in 0.12 us whatever its size, so two warps copy rows of 2,048 columns, and
// narrower ones come by 16-byte asynchronous copies of six warps.
//
// What bounds it, us per step, single launches / loop (logistic, N workers, B rows): 32 workers, d = 8,192, B = 256 50.4 / 47.7, of which 41 are the
// rows at the copy rate, the rest the end of a step, less what the ring holds (192 KB per CTA); 8 workers, d = 8,192, B = 256 46.0 / 25.7, the
// chain of a group and the ring; 8 workers, d = 752, B = 256 47.2 / 9.4, eight groups and the end of a step (4); 4 workers, d = 64, B = 100
// 22.5 / 6.6; 16 workers, d = 8,216, B = 16 23.4 / 9.0.  Tried: the end of a step by the warps of u (44 to 130 us at the first shape: spilled
// registers), rows two groups ahead in registers (55.3: the same), the next rows prefetched to L2 while a step ends (48.0 to 49.3).
// 96 registers per thread do not hold this form's values either: 24 to 132 bytes of spill stores per thread with fixed widths (76 in the kernel of the first
// shape), 114 to 166 with the others.
//
// Arithmetic, operation for operation, is that of the per-step kernels.
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "lpc_device.cuh"
#include "lpc_inner.h"
#include "lpc_words.cuh"

namespace cg = cooperative_groups;

namespace lpc {
namespace {

constexpr int LCS = 8;         // CTAs per cluster at most
constexpr int LSLOTS = 16;     // exchange slots for margin partial sums
constexpr int LMAXR = 8;       // ring stages at most
constexpr int LMAXB = 256;     // rows per worker
constexpr int LMAXN = 64;      // workers
constexpr int LFLAGS = 256;    // scale words of a parity half
constexpr int LPUB = 16;       // scale words sit 128 bytes apart
constexpr int DW = 8, KW = 2;  // warps: margins (two sides of four) and the end of a step, coefficients
constexpr int DT = DW * 32;

// NB: blocks of 128 columns per slice.
template <int NB>
struct Shape {
  static constexpr int SL = 128 * NB;
  static constexpr int QB = NB < 4 ? NB : 4;        // blocks per margin warp
  static constexpr int CP = NB / QB;                // column parts of a slice
  static constexpr int RP = 4 / CP;                 // row parts of a group
  static constexpr int V = NB >= 2 ? 16 : 8;        // (row, block) pairs per margin warp: one reduction
  static constexpr int RW = V / QB;                 // rows per margin warp
  static constexpr int GR = RP * RW;                // rows per group: 4, 8, 16, 32, 32
  static constexpr bool BULK = NB == 16, AHEAD = NB == 16;
  static constexpr int UW = NB == 16 ? 8 : 4;       // warps that own the coordinates of u
  static constexpr int EU = SL / (UW * 32);         // coordinates per thread: pieces of at most four, `APART` apart
  static constexpr int PE = EU < 4 ? EU : 4, PIECES = EU / PE, APART = UW * 128;
  static constexpr int REFILL = BULK ? 2 : 6;       // warps
  static constexpr int W_U = DW, W_K = W_U + UW, W_REFILL = W_K + KW;
  static constexpr int NT = (W_REFILL + REFILL) * 32;  // 20 warps: 96 registers per thread
  static constexpr size_t STAGE = (size_t)GR * SL * 4;
};

struct LSmem {
  uint64_t sbar[LMAXR];   // stage filled
  uint64_t ebar[LMAXR];   // stage read
  uint64_t pbar[LSLOTS];  // a group's margin partial sums have arrived from every CTA
  uint64_t cbar[LSLOTS];  // its coefficients are in `coefs`
  uint64_t ibar[2];       // sampled rows of a step (by parity)
  uint64_t mbar[2];       // their labels and snapshot sides
  uint64_t ubar;          // the step's u is in `us`
  unsigned long long sx[2][3 * LCS];  // statistics of every CTA of the cluster: tagged words, written by the peers
  __align__(16) float coefs[LSLOTS][32];
  float ws1[DW], ws2[DW];
  uint32_t wmax[DW], wclip[DW];
  Scale scale;
  int failed;
};

__device__ __forceinline__ void sync_ends() { asm volatile("bar.sync 1, 256;" ::: "memory"); }  // the warps that end a step
static_assert(DT == 256, "sync_ends");

__device__ __noinline__ Scale scale_of(uint32_t max_bits, float S1, float S2, ScaleRule rule, int b, int clip_mode, float clip_value) {
  return make_scale_in_loop(max_bits, S1, S2, rule, b, clip_mode, clip_value);
}
// Step 6 of Algorithm 2: x = tau1 z + tau2 x~ + (1 - tau1 - tau2) y.
__device__ __forceinline__ float couple(const PersistArgs& pa, float z, float xt, float y) {
  const float tau3 = __fsub_rn(__fsub_rn(1.0f, pa.tau1), pa.tau2);
  return add_rn(add_rn(mul_rn(pa.tau1, z), mul_rn(pa.tau2, xt)), mul_rn(tau3, y));
}

// The end of a step, by the margin warps, which have nothing else to do then: statistics, scale, codes and their words, the other workers'
// words, the new point in `xs`.  (By the warps of u the step's end took registers from their loop over the groups of rows: values spilled to
// local memory, which has next to no first-level cache beside this much shared memory.)
template <int BITS, int NB, bool ALPC>
__device__ __forceinline__ void end_of_step(const PersistArgs& pa, float* ring, float* xs, const float* us, LSmem& sm, int t, float wcur) {
  constexpr int SL = Shape<NB>::SL;
  const InnerArgs& a = pa.in;
  const int d = a.d, N = a.N, CW = a.CS, b = BITS ? BITS : a.b;
  float* state = xs + SL;
  const int tu = threadIdx.x, lane = tu & 31, wu = tu >> 5;
  const int rank = (int)cg::this_cluster().block_rank(), worker = blockIdx.y, c0 = rank * SL;
  const bool is_J = ALPC && worker == N;
  const int off8 = tu * 8, c = c0 + off8;        // this thread's eight coordinates from the scale on
  const bool mine = off8 < SL && c < d;
  const float invN = __fdiv_rn(1.0f, (float)N), invB = __fdiv_rn(1.0f, (float)a.B);
  const float kappa = mul_rn(pa.eta, pa.lambda_l1), kappa_y = mul_rn(pa.inv4L, pa.lambda_l1), kappa_z = mul_rn(pa.alpha, pa.lambda_l1);
  constexpr int WPG = BITS == 0 ? 8 : (BITS == 8 ? 2 : 1);  // tagged words per group of 8 coordinates, at most
  const int wpg = BITS == 0 ? pa.wpg : WPG;
  const size_t groups = (size_t)(CW * SL) >> 3;
  auto expired = [&](uint32_t it, uint64_t& t0) -> bool {
    if ((it & 63u) != 63u) return false;
    return spin_expired(it, t0, pa.abort_flag, a.dev_status);
  };
  const uint64_t k = a.k_base + (uint64_t)t;
  const int wpar = (pa.count - 1 - t) & 1;
  const bool last = t == pa.count - 1;
  const uint32_t tag = pa.tag_base + (uint32_t)(t + 1);
  float xo[8], u[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) xo[e] = off8 < SL ? xs[off8 + e] : 0.f;
  U4 rnd = U4{0, 0, 0, 0};
  if (b != 32) rnd = stream_block(a.seed, TAG_ROUND, (uint32_t)worker, k, (uint32_t)(c >> 3));
#pragma unroll
  for (int e = 0; e < 8; ++e) u[e] = off8 < SL ? mul_rn(us[off8 + e], invB) : 0.f;

  if (is_J) {  // step 11 of Algorithm 2: v^ = u_J + mu in full precision
    if (off8 < SL) {
      unsigned long long* q = pa.ll_vhat + (size_t)wpar * groups * 8 + c;
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        const float v0 = add_rn(u[e], c + e < d ? a.mu[c + e] : 0.f), v1 = add_rn(u[e + 1], c + e + 1 < d ? a.mu[c + e + 1] : 0.f);
        st_word2(q + e, __float_as_uint(v0), __float_as_uint(v1), tag);
        if (last && c + e < d) pa.vhat[c + e] = v0;
        if (last && c + e + 1 < d) pa.vhat[c + e + 1] = v1;
      }
    }
  } else {
    // scale (Eq. 2)
    uint32_t mx = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) mx = max(mx, __float_as_uint(fabsf(u[e])));
    if (a.clip_mode == CLIP_STD) {
      float sq[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) sq[e] = mul_rn(u[e], u[e]);
      const float s1 = warp_tree_sum(tree8(u)), s2 = warp_tree_sum(tree8(sq));
      if (lane == 0) { sm.ws1[wu] = s1; sm.ws2[wu] = s2; }
    }
    mx = warp_max_u32(mx);
    if (lane == 0) sm.wmax[wu] = mx;
    sync_ends();
    if (wu == 0) {  // lane 8 k + i, k = 0, 1, 2 for max |u|, S1, S2: the CTA's from those of warp i, then the rank i's
      const int kk = lane >> 3, i = lane & 7;
      auto join = [&](uint32_t x, uint32_t y) { return kk == 0 ? max(x, y) : __float_as_uint(add_rn(__uint_as_float(x), __uint_as_float(y))); };
      auto join_lanes = [&](uint32_t v) {
#pragma unroll
        for (int m = 1; m < 8; m <<= 1) v = join(v, __shfl_xor_sync(0xFFFFFFFFu, v, m));
        return v;
      };
      const bool sums = a.clip_mode == CLIP_STD;
      uint32_t v = kk == 0 ? sm.wmax[i] : sums ? __float_as_uint(kk == 1 ? sm.ws1[i] : sm.ws2[i]) : 0u;
      v = join_lanes(v);
      if (CW > 1) {
        const bool sends = kk < 3 && i < CW;
        if (sends) st_cluster_word(&sm.sx[t & 1][kk * LCS + rank], (uint32_t)i, v, tag);
        uint64_t t0 = 0;
        v = 0u;  // slices without a column add zeros
        for (uint32_t it = 0;; ++it) {
          bool ok = true;
          if (sends) {
            const unsigned long long w = ld_shared_word(&sm.sx[t & 1][kk * LCS + i]);
            ok = word_tag(w) == tag;
            v = (uint32_t)w;
          }
          if (__all_sync(0xFFFFFFFFu, ok) || __any_sync(0xFFFFFFFFu, expired(it, t0))) break;
        }
        v = join_lanes(v);
      }
      const uint32_t m = __shfl_sync(0xFFFFFFFFu, v, 0);
      const float S1 = __uint_as_float(__shfl_sync(0xFFFFFFFFu, v, 8)), S2 = __uint_as_float(__shfl_sync(0xFFFFFFFFu, v, 16));
      const Scale own = scale_of(m, S1, S2, pa.rule, b, a.clip_mode, a.clip_value);
      if (lane == 0) {
        sm.scale = own;
        st_word(pa.pub + ((size_t)wpar * LFLAGS + worker * CW + rank) * LPUB, __float_as_uint(own.delta), tag);
        if (rank == 0) {
          if (last) a.delta[worker] = own.delta;
          if (own.flags & 2u) atomicOr(a.dev_status, DEV_NONFINITE);
        }
      }
    }
    sync_ends();
    const Scale sc = sm.scale;
    const bool degenerate = (sc.flags & 1u) != 0;
    const uint32_t zero_code = (b == 1) ? 0u : (1u << (b - 1));
    uint32_t* out = a.codes + (int64_t)worker * a.stride_words;
    unsigned long long* q = pa.ll + (((size_t)wpar * N + worker) * groups + (size_t)(c >> 3)) * wpg;
    uint32_t nclip = 0;
    uint64_t lo = 0, hi = 0;
    if (b == 32) {
      if (off8 < SL) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          float v = u[e];
          if (a.clip_mode != CLIP_NONE && c + e < d) {
            if (v > sc.T) { v = sc.T; ++nclip; }
            if (v < -sc.T) { v = -sc.T; ++nclip; }
          }
          const uint32_t bits = c + e < d ? __float_as_uint(v) : 0u;
          st_word(q + e, bits, tag);
          if (last && c + e < a.pad_words) out[c + e] = bits;
        }
      }
    } else if (mine) {
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        if (c + e < d) {
          uint32_t code = zero_code;
          if (!degenerate) {
            const uint32_t r16 = lane16(rnd, e);
            code = BITS ? quantize_code<BITS ? BITS : 2>(u[e], sc.rdelta, r16) : quantize_code_rt(u[e], sc.rdelta, r16, b);
            nclip += (u[e] > sc.T || u[e] < sc.lower) ? 1u : 0u;
          }
          const int pos = e * b;
          if (pos < 64) {
            lo |= (uint64_t)code << pos;
            if (pos + b > 64) hi |= (uint64_t)code >> (64 - pos);
          } else {
            hi |= (uint64_t)code << (pos - 64);
          }
        }
      }
    }
    if (b != 32 && off8 < SL) {
      if constexpr (BITS == 8) {
        st_word2(q, (uint32_t)lo, (uint32_t)(lo >> 32), tag);
      } else {
        st_word(q, (uint32_t)lo, tag);
        if (BITS == 0 && wpg >= 2) st_word(q + 1, (uint32_t)(lo >> 32), tag);
      }
      if (BITS == 0 && wpg >= 4) {
        st_word(q + 2, (uint32_t)hi, tag);
        st_word(q + 3, (uint32_t)(hi >> 32), tag);
      }
    }
    if (last) {  // the caller's copy of the last messages, and their counts
      if (b != 32) {
        if constexpr (BITS == 8 || BITS == 4) {
          const int64_t w = ((int64_t)c * BITS) >> 5;
          if (off8 < SL && w < a.pad_words) {
            out[w] = (uint32_t)lo;
            if (BITS == 8) out[w + 1] = (uint32_t)(lo >> 32);  // pad_words is a multiple of 4
          }
        } else if constexpr (BITS == 2 || BITS == 1) {
          constexpr int LPS = 4 / BITS;  // lanes per word of the stream
          uint32_t word = (uint32_t)lo;
#pragma unroll
          for (int i = 1; i < LPS; ++i) word |= __shfl_down_sync(0xFFFFFFFFu, (uint32_t)lo, i) << (i * 8 * BITS);
          const int64_t w = ((int64_t)c * BITS) >> 5;
          if (off8 < SL && (lane & (LPS - 1)) == 0 && w < a.pad_words) out[w] = word;
        } else {  // through the ring, which nobody reads any more: every group has been taken
          uint8_t* stage = reinterpret_cast<uint8_t*>(ring);
          for (int i = 0; i < b; ++i) stage[tu * b + i] = (uint8_t)((i < 8) ? (lo >> (8 * i)) : (hi >> (8 * (i - 8))));
          sync_ends();
          const int64_t w0 = (int64_t)(c0 >> 5) * b;
          for (int w = tu; w < (SL / 32) * b; w += DT)
            if (w0 + w < a.pad_words) out[w0 + w] = reinterpret_cast<const uint32_t*>(stage)[w];
        }
      }
      nclip = __reduce_add_sync(0xFFFFFFFFu, nclip);
      if (lane == 0) sm.wclip[wu] = nclip;
      sync_ends();
      if (tu == 0) {
        uint32_t n = 0;
        for (int w = 0; w < DW; ++w) n += sm.wclip[w];
        a.clipped_part[worker * LCS + rank] = clipped_word(n, CW);
      }
    }
  }

  // x_{t+1} from the words of all workers (Eq. 3, the proximal step; Algorithm 2: steps 12, 13 and the next step 6)
  float acc[8];
  f32x2 acc2[4];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) acc2[e] = 0ull;
  float muv[8];
#pragma unroll
  for (int e = 0; e < 8; e += 4) {  // d is a multiple of 4
    const float4 r = off8 < SL && c + e < d ? *reinterpret_cast<const float4*>(a.mu + c + e) : make_float4(0.f, 0.f, 0.f, 0.f);
    muv[e] = r.x; muv[e + 1] = r.y; muv[e + 2] = r.z; muv[e + 3] = r.w;
  }
  const unsigned long long* dwords = pa.pub + ((size_t)wpar * LFLAGS + rank) * LPUB;
  const unsigned long long* from = pa.ll + ((size_t)wpar * N * groups + (mine ? (size_t)(c >> 3) : (size_t)(c0 >> 3))) * wpg;
  // one round: the words of `CHW` workers, W each, and their scales in flight together; add(worker of the round, its scale, its words)
  auto rounds = [&](auto words, auto per_round, auto&& add) {
    constexpr int W = decltype(words)::value, CHW = decltype(per_round)::value;
#pragma unroll 1
    for (int i0 = 0; i0 < N; i0 += CHW) {
      unsigned long long cw[CHW][W], dw;
      uint64_t t0 = 0;
      const int his = i0 + (lane & (CHW - 1));  // the worker whose scale this lane fetches
#pragma unroll 1
      for (uint32_t it = 0;; ++it) {
        dw = ld_word(dwords + (size_t)min(his, N - 1) * CW * LPUB);
        bool ok = word_tag(dw) == tag;
#pragma unroll
        for (int j = 0; j < CHW; ++j) ld_words<W>(from + (size_t)min(i0 + j, N - 1) * groups * W, cw[j]);
#pragma unroll
        for (int j = 0; j < CHW; ++j)
#pragma unroll
          for (int w = 0; w < W; ++w) ok = ok && word_tag(cw[j][w]) == tag;
        if (__all_sync(0xFFFFFFFFu, ok) || __any_sync(0xFFFFFFFFu, expired(it, t0))) break;
      }
      const uint32_t dmine = his < N ? (uint32_t)dw : 0u;
#pragma unroll
      for (int j = 0; j < CHW; ++j) {
        const float di = __uint_as_float(__shfl_sync(0xFFFFFFFFu, dmine, j));
        if (i0 + j < N) add(di, cw[j]);
      }
    }
  };
  if constexpr (BITS != 0) {
    rounds(std::integral_constant<int, WPG>(), std::integral_constant<int, 16 / WPG>(), [&](float di, const unsigned long long (&cw)[WPG]) {
      uint64_t l = (uint32_t)cw[0];
      if constexpr (WPG >= 2) l |= (uint64_t)(uint32_t)cw[1] << 32;
      f32x2 k2[4];
      decode_pairs<BITS ? BITS : 1, 8>(l, k2);
#pragma unroll
      for (int e = 0; e < 4; ++e) acc2[e] = add_scaled_pair<BITS>(acc2[e], pack2(di, di), k2[e]);
    });
  } else {
    // The width decides how many words a group has.  One loop for all widths fetched eight words of four workers one by one: every sector came
    // once per word, and values spilled.  Sixteen words a round in whole accesses, us per step before / after: b = 12, 32 workers, d = 2,432,
    // B = 128 43.7 / 36.7; b = 16, 16 workers, d = 4,896, B = 100 30.8 / 26.6; b = 32, 16 workers, d = 5,156, B = 200 53.0 / 40.7; b = 32, 32 workers,
    // d = 4,000, B = 66 40.5 / 26.5.  Tried: the step's end as a function of its own (1.17 to 1.33 times as long), the snapshot gradient and the old
    // point read after the rounds (fewer spills, 0.95 to 1.05 times).
    const uint32_t mask = b < 32 ? (1u << b) - 1u : 0u;
    auto add_index = [&](int e, float di, uint32_t code) { acc[e] = add_scaled_index<0>(acc[e], di, index_as_float(code, b)); };
    if (wpg == 1) {
      rounds(std::integral_constant<int, 1>(), std::integral_constant<int, 16>(), [&](float di, const unsigned long long (&cw)[1]) {
#pragma unroll
        for (int e = 0; e < 8; ++e) add_index(e, di, ((uint32_t)cw[0] >> (e * b)) & mask);
      });
    } else if (wpg == 2) {
      rounds(std::integral_constant<int, 2>(), std::integral_constant<int, 8>(), [&](float di, const unsigned long long (&cw)[2]) {
        const uint64_t l = (uint32_t)cw[0] | (uint64_t)(uint32_t)cw[1] << 32;
#pragma unroll
        for (int e = 0; e < 8; ++e) add_index(e, di, (uint32_t)(l >> (e * b)) & mask);
      });
    } else if (wpg == 4) {
      rounds(std::integral_constant<int, 4>(), std::integral_constant<int, 4>(), [&](float di, const unsigned long long (&cw)[4]) {
        const uint64_t l = (uint32_t)cw[0] | (uint64_t)(uint32_t)cw[1] << 32, h = (uint32_t)cw[2] | (uint64_t)(uint32_t)cw[3] << 32;
#pragma unroll
        for (int e = 0; e < 8; ++e) add_index(e, di, extract_bits(l, h, e * b, b));
      });
    } else {
      rounds(std::integral_constant<int, 8>(), std::integral_constant<int, 2>(), [&](float di, const unsigned long long (&cw)[8]) {
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[e] = add_rn(acc[e], mul_rn(di, c + e < d ? __uint_as_float((uint32_t)cw[e]) : 0.f));
      });
    }
  }
  if constexpr (BITS != 0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) unpack2(acc2[e], acc[2 * e], acc[2 * e + 1]);
  }
  unsigned long long vw[ALPC ? 8 : 1];
  if constexpr (ALPC) {
    uint64_t t0 = 0;
    const unsigned long long* q = pa.ll_vhat + (size_t)wpar * groups * 8 + (mine ? c : c0);
#pragma unroll 1
    for (uint32_t it = 0;; ++it) {
      bool ok = true;
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        ld_word2(q + e, vw[e], vw[e + 1]);
        ok = ok && word_tag(vw[e]) == tag && word_tag(vw[e + 1]) == tag;
      }
      if (ok || expired(it, t0)) break;
    }
  }
  if (off8 < SL) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float x = 0.f;
      if (c + e < d) {
        const float v = add_rn(mul_rn(acc[e], invN), muv[e]);
        if constexpr (ALPC) {
          const float vhat = __uint_as_float((uint32_t)vw[e]);
          const float yn = mul_rn(soft_threshold(__fsub_rn(xo[e], mul_rn(pa.inv4L, v)), kappa_y), pa.cy);
          const float zn = mul_rn(soft_threshold(__fsub_rn(state[SL + off8 + e], mul_rn(pa.alpha, vhat)), kappa_z), pa.cz);
          const float sn = add_rn(state[2 * SL + off8 + e], mul_rn(wcur, yn));
          state[off8 + e] = yn;
          state[SL + off8 + e] = zn;
          state[2 * SL + off8 + e] = sn;
          x = last ? xo[e] : couple(pa, zn, pa.xt[c + e], yn);  // the coupled point of the last step stays
          if (last && worker == 0) { pa.y[c + e] = yn; pa.z[c + e] = zn; pa.ysum[c + e] = sn; }
        } else {
          x = soft_threshold(__fsub_rn(xo[e], mul_rn(pa.eta, v)), kappa);
        }
        if (last && worker == 0) pa.x_out[c + e] = x;
      }
      xs[off8 + e] = x;  // the margins of this step are all formed: nobody reads the old point any more but its owner here
    }
  }
}

template <int BITS, int NB, bool ALPC>
__global__ void __launch_bounds__(Shape<NB>::NT, 1) stream_loop_kernel(const __grid_constant__ PersistArgs pa) {
  using S = Shape<NB>;
  constexpr int SL = S::SL, GR = S::GR, CP = S::CP, QB = S::QB, RW = S::RW;
  const InnerArgs& a = pa.in;
  cg::cluster_group cluster = cg::this_cluster();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int R = a.stream_stages, B = a.B, d = a.d, N = a.N, CW = a.CS, Bp = (B + 3) & ~3;
  float* ring = reinterpret_cast<float*>(smem_raw);
  float* xs = ring + (size_t)R * GR * SL;              // the step's point
  float* state = xs + SL;                              // ALPC: y, z, sum of y
  float* us = state + (ALPC ? 3 * SL : 0);             // the step's u on its way from the warps that add it up
  float* parts = us + SL;                              // [slot][(CTA * CP + part) * GR + row]
  int64_t* idx = reinterpret_cast<int64_t*>(parts + (size_t)LSLOTS * GR * CP * CW);
  float* yv = reinterpret_cast<float*>(idx + 2 * Bp);
  float* ms = yv + 2 * Bp;
  LSmem& sm = *reinterpret_cast<LSmem*>(ms + 2 * Bp);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster.block_rank(), worker = blockIdx.y;
  const bool is_J = ALPC && worker == N;
  const int c0 = rank * SL, width = min(SL, d - c0);   // > 0: a cluster has as many CTAs as there are slices with columns
  const int ng = (B + GR - 1) / GR, total = pa.count * ng;

  if (tid < LMAXR) {
    mbar_init(&sm.sbar[tid], S::BULK ? S::REFILL : S::REFILL * 32);
    mbar_init(&sm.ebar[tid], S::UW + DW / 2);
  } else if (tid < LMAXR + LSLOTS) {
    mbar_init(&sm.pbar[tid - LMAXR], 1);
    mbar_init(&sm.cbar[tid - LMAXR], 1);
  } else if (tid < LMAXR + LSLOTS + 2) {
    mbar_init(&sm.ibar[tid - LMAXR - LSLOTS], S::UW);
    mbar_init(&sm.mbar[tid - LMAXR - LSLOTS], S::UW);
  } else if (tid == LMAXR + LSLOTS + 2) {
    mbar_init(&sm.ubar, S::UW);
    sm.failed = 0;
  }
  if (tid < 32) mbar_fence_init();
  if (tid >= 64 && tid < 64 + 2 * 3 * LCS) (&sm.sx[0][0])[tid - 64] = 0ull;  // tags start at 1
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  bool gave_up = false;  // after one wait ran out this thread waits no more (the status word says so)
  auto wait_on = [&](uint64_t* bar, uint32_t parity, bool from_cluster = false) {
    if (gave_up) return;
    if (!from_cluster && mbar_test(bar, parity)) return;
    if (!(from_cluster ? mbar_wait_cluster(bar, parity) : mbar_wait(bar, parity))) {
      atomicOr(a.dev_status, DEV_TIMEOUT);
      sm.failed = 1;
      gave_up = true;
    }
  };
  struct Ring {  // stage and phase of the group that a warp is at
    int s = 0;
    uint32_t parity = 0;
    __device__ __forceinline__ void advance(int R) {
      if (++s == R) { s = 0; parity ^= 1u; }
    }
  };

  if (warp < DW) {
    // ---- margins: the four warps of a side share a group, the sides take the groups of the even and of the odd stages (each then sees
    // every phase of its stages).  Warp w of a side takes QB blocks of 128 columns of RW rows; lane l the columns 128 q + 4 l .. + 3.
    const int side = warp >> 2, cp = (warp & 3) % CP, rp = (warp & 3) / CP;
    constexpr int LOGV = S::V == 16 ? 4 : 3, LOGR = RW == 8 ? 3 : 2;
    static_assert((1 << LOGR) == RW && (1 << LOGV) == S::V, "rows and pairs per warp");
    const int myrow = rp * RW + halving_index<LOGR>(lane);
    {  // the first step's point
      const int off8 = tid * 8, c = c0 + off8;
      if (off8 < SL) {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const bool in = c + e < d;
          float x = 0.f;
          if constexpr (ALPC) {
            const float y0 = in ? pa.y[c + e] : 0.f, z0 = in ? pa.z[c + e] : 0.f;
            state[off8 + e] = y0;
            state[SL + off8 + e] = z0;
            state[2 * SL + off8 + e] = in ? pa.ysum[c + e] : 0.f;
            if (in) x = couple(pa, z0, pa.xt[c + e], y0);
          } else {
            if (in) x = a.x[c + e];
          }
          xs[off8 + e] = x;
        }
      }
    }
    Ring at;
    int gg = 0;
    float wcur = pa.w0;  // snapshot weight of the step
#pragma unroll 1
    for (int t = 0; t < pa.count; ++t) {
      sync_ends();
      float4 xv[QB];
#pragma unroll
      for (int q = 0; q < QB; ++q) {
        const int off = (cp * QB + q) * 128 + lane * 4;  // width is a multiple of 4
        xv[q] = off < width ? *reinterpret_cast<const float4*>(xs + off) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll 1
      for (int g = 0; g < ng; ++g, ++gg, at.advance(R)) {
        if ((at.s & 1) != side) continue;
        wait_on(&sm.sbar[at.s], at.parity);
        const float* src = ring + (size_t)(at.s * GR + rp * RW) * SL + cp * QB * 128 + lane * 4;
        float sv[S::V];
        auto products = [&](auto whole) {
#pragma unroll
          for (int h = 0; h < RW; h += 2) {  // two rows at a time
            float4 v[2][QB];
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
              for (int q = 0; q < QB; ++q)
                v[j][q] = decltype(whole)::value || (cp * QB + q) * 128 + lane * 4 < width
                              ? *reinterpret_cast<const float4*>(src + (h + j) * SL + q * 128) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int j = 0; j < 2; ++j)
#pragma unroll
              for (int q = 0; q < QB; ++q) {
                float p0, p1, p2, p3;
                unpack2(mul2_rn(pack2(v[j][q].x, v[j][q].y), pack2(xv[q].x, xv[q].y)), p0, p1);
                unpack2(mul2_rn(pack2(v[j][q].z, v[j][q].w), pack2(xv[q].z, xv[q].w)), p2, p3);
                sv[(h + j) * QB + q] = tree4(p0, p1, p2, p3);
              }
          }
        };
        if (width == SL) products(std::true_type());  // the usual case: nothing to test per load
        else products(std::false_type());
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.ebar[at.s]);
        WarpHalving<S::V, 0>::run(sv, lane);  // lane holds the 32-lane tree sum of (row, block) halving_index<LOGV>(lane)
        float part = sv[0];
#pragma unroll
        for (int m = S::V / 2; m >= RW; m >>= 1) part = add_rn(part, __shfl_xor_sync(0xFFFFFFFFu, part, m));  // the tree over the blocks
        const int sl = gg % LSLOTS;
        if (myrow < B - g * GR) {
          for (int q = lane / RW; q < CW; q += 32 / RW)
            st_async_cluster(&parts[((size_t)sl * CW * CP + rank * CP + cp) * GR + myrow], &sm.pbar[sl], (uint32_t)q, __float_as_uint(part));
        }
      }
      wait_on(&sm.ubar, (uint32_t)(t & 1));
      end_of_step<BITS, NB, ALPC>(pa, ring, xs, us, sm, t, wcur);
      if constexpr (ALPC) wcur = mul_rn(wcur, pa.theta);
    }
  } else if (warp < S::W_K) {
    // ---- u -----------------------------------------------------------------------------------------------------------------------
    const int tu = tid - S::W_U * 32;
    // the rows of a step, their labels and the snapshot side of their coefficients: for the first two steps now, for the others two steps
    // ahead, when a step's u has been handed over (all of its rows have been used by then, and nothing else is to be done here)
    const int64_t span = (a.sample_global || is_J) ? a.n : a.n / N, first = (a.sample_global || is_J) ? 0 : (int64_t)worker * span;
    auto draw = [&](int t) {
      const int half = (t & 1) * Bp;
#pragma unroll 1
      for (int slot = tu; slot < B; slot += S::UW * 32) {
        const U4 r = stream_block(a.seed, is_J ? TAG_BATCH_J : TAG_BATCH, is_J ? 0u : (uint32_t)worker, a.k_base + (uint64_t)t, (uint32_t)slot);
        idx[half + slot] = first + (int64_t)(((uint64_t)r.x * (uint64_t)span) >> 32);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.ibar[t & 1]);
#pragma unroll 1
      for (int slot = tu; slot < B; slot += S::UW * 32) {
        const int64_t row = idx[half + slot];
        const float y = a.y[row];
        yv[half + slot] = y;
        ms[half + slot] = loss_deriv(a.loss, a.margins[row], y);
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.mbar[t & 1]);
    };
    draw(0);
    if (pa.count > 1) draw(1);
    float ua[S::EU];
#pragma unroll
    for (int e = 0; e < S::EU; ++e) ua[e] = 0.f;
    // this thread's values of row j of a stage (rows past a ragged end are read and not used)
    auto row = [&](const float* src, int j, float* v, auto whole) {
#pragma unroll
      for (int p = 0; p < S::PIECES; ++p) {
        const bool in = decltype(whole)::value || p * S::APART + tu * S::PE < width;
        if constexpr (S::PE == 4) {
          const float4 r = in ? *reinterpret_cast<const float4*>(src + j * SL + p * S::APART) : make_float4(0.f, 0.f, 0.f, 0.f);
          v[p * 4] = r.x; v[p * 4 + 1] = r.y; v[p * 4 + 2] = r.z; v[p * 4 + 3] = r.w;
        } else if constexpr (S::PE == 2) {
          const float2 r = in ? *reinterpret_cast<const float2*>(src + j * SL) : make_float2(0.f, 0.f);
          v[0] = r.x; v[1] = r.y;
        } else {
          v[0] = in ? src[j * SL] : 0.f;
        }
      }
    };
    auto add_row = [&](float cf, const float* v) {
      if constexpr (S::EU == 1) {
        ua[0] = add_rn(ua[0], mul_rn(cf, v[0]));
      } else {
#pragma unroll
        for (int e = 0; e < S::EU; e += 2) {  // products in pairs, sums one by one: ptxas may join a product and a sum of pairs
          float p0, p1;
          unpack2(mul2_rn(pack2(cf, cf), pack2(v[e], v[e + 1])), p0, p1);
          ua[e] = add_rn(ua[e], p0);
          ua[e + 1] = add_rn(ua[e + 1], p1);
        }
      }
    };
    auto give_back = [&](int s) {
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.ebar[s]);
    };
    // AHEAD: a group's rows go into registers before its coefficients are there, so that its stage goes back at once; narrower slices have
    // the whole minibatch or much of it in the ring anyway
    Ring at;
    int t = 0, g = 0;
#pragma unroll 1
    for (int gg = 0; gg < total; ++gg) {
      const int cnt = min(GR, B - g * GR), sl = gg % LSLOTS;
      if constexpr (S::AHEAD) {
        float v[GR][S::EU];
        wait_on(&sm.sbar[at.s], at.parity);
        const float* src = ring + (size_t)at.s * GR * SL + tu * S::PE;
        if (width == SL) {
#pragma unroll
          for (int j = 0; j < GR; ++j) row(src, j, v[j], std::true_type());
        } else {
#pragma unroll
          for (int j = 0; j < GR; ++j) row(src, j, v[j], std::false_type());
        }
        give_back(at.s);
        wait_on(&sm.cbar[sl], (uint32_t)((gg / LSLOTS) & 1));
        const float4 c4 = *reinterpret_cast<const float4*>(sm.coefs[sl]);
        const float cj[4] = {c4.x, c4.y, c4.z, c4.w};
        static_assert(!S::AHEAD || GR == 4, "one vector of coefficients");
        if (cnt == GR) {
#pragma unroll
          for (int j = 0; j < 4; ++j) add_row(cj[j], v[j]);
        } else {
#pragma unroll
          for (int j = 0; j < 3; ++j)
            if (j < cnt) add_row(cj[j], v[j]);
        }
      } else {
        wait_on(&sm.sbar[at.s], at.parity);
        wait_on(&sm.cbar[sl], (uint32_t)((gg / LSLOTS) & 1));
        const float* src = ring + (size_t)at.s * GR * SL + tu * S::PE;
        auto rows4 = [&](int j0, auto whole) {
          float v[4][S::EU];
#pragma unroll
          for (int j = 0; j < 4; ++j) row(src, j0 + j, v[j], whole);
          const float4 c4 = *reinterpret_cast<const float4*>(&sm.coefs[sl][j0]);
          const float cj[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j0 + j < cnt) add_row(cj[j], v[j]);
        };
        if (width == SL) {
#pragma unroll 2
          for (int j0 = 0; j0 < GR; j0 += 4) rows4(j0, std::true_type());
        } else {
#pragma unroll 2
          for (int j0 = 0; j0 < GR; j0 += 4) rows4(j0, std::false_type());
        }
        give_back(at.s);
      }
      at.advance(R);
      if (++g < ng) continue;

      // the end of step t: u to the warps that go on with it
      g = 0;
#pragma unroll
      for (int p = 0; p < S::PIECES; ++p)
#pragma unroll
        for (int e = 0; e < S::PE; ++e) us[p * S::APART + tu * S::PE + e] = ua[p * S::PE + e];
#pragma unroll
      for (int e = 0; e < S::EU; ++e) ua[e] = 0.f;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.ubar);
      if (t + 2 < pa.count) draw(t + 2);
      ++t;
    }
  } else if (warp < S::W_REFILL) {
    // ---- coefficients (warp c of these takes the groups c, c + KW, ...) ---------------------------------------------------------
    constexpr int LR = GR < 32 ? GR : 32, LQ = 32 / LR, QL = LCS / LQ;  // rows and ranges of CTAs side by side in a warp, CTAs per lane
    const int j = lane % LR, q0 = (lane / LR) * QL;
    int t = 0, g = warp - S::W_K;
    while (g >= ng) { g -= ng; ++t; }
#pragma unroll 1
    for (int gg = warp - S::W_K; gg < total; gg += KW) {
      const int cnt = min(GR, B - g * GR), sl = gg % LSLOTS, half = t & 1;
      if (lane == 0) mbar_expect_tx(&sm.pbar[sl], (uint32_t)(CW * cnt * CP * 4));
      __syncwarp();
      wait_on(&sm.mbar[half], (uint32_t)((t >> 1) & 1));
      wait_on(&sm.pbar[sl], (uint32_t)((gg / LSLOTS) & 1), true);
      float mq[QL];
#pragma unroll
      for (int i = 0; i < QL; ++i) {  // the tree over the parts of a slice; slices without a column add zeros
        const float* p = parts + ((size_t)sl * CW * CP + (size_t)(q0 + i) * CP) * GR + j;
        mq[i] = 0.f;
        if (q0 + i < CW && j < cnt) {
          if constexpr (CP == 4) mq[i] = tree4(p[0], p[GR], p[2 * GR], p[3 * GR]);
          else if constexpr (CP == 2) mq[i] = add_rn(p[0], p[GR]);
          else mq[i] = p[0];
        }
      }
      float m = mq[0];
      if constexpr (QL >= 2) {
        if (CW > 1) m = add_rn(mq[0], mq[1]);
      }
      if constexpr (QL >= 4) {
        if (CW > 2) m = add_rn(m, add_rn(mq[2], mq[3]));
      }
      if constexpr (QL >= 8) {
        if (CW > 4) m = add_rn(m, tree4(mq[4], mq[5], mq[6], mq[7]));
      }
#pragma unroll
      for (int x = LR, n = QL; x < 32; x <<= 1, n <<= 1)
        if (CW > n) m = add_rn(m, __shfl_xor_sync(0xFFFFFFFFu, m, x));
      if (lane < LR) {
        float cf = 0.f;
        if (j < cnt) {
          const int slot = g * GR + j;
          cf = __fsub_rn(loss_deriv(a.loss, m, yv[half * Bp + slot]), ms[half * Bp + slot]);
          if (rank == 0 && t == pa.count - 1) {
            if (a.idx_tap) a.idx_tap[(int64_t)worker * B + slot] = idx[half * Bp + slot];
            if (a.coef_tap) a.coef_tap[(int64_t)worker * B + slot] = cf;
          }
        }
        sm.coefs[sl][j] = cf;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.cbar[sl]);
      g += KW;
      while (g >= ng) { g -= ng; ++t; }
    }
  } else {
    // ---- refills: a stage is filled again the moment it has been handed over, with rows of the next step where this one's are through ---
    const int wr = warp - S::W_REFILL;
    Ring at;
    int gg = 0;
#pragma unroll 1
    for (int t = 0; t < pa.count; ++t) {
      wait_on(&sm.ibar[t & 1], (uint32_t)((t >> 1) & 1));
      const int64_t* rows = idx + (t & 1) * Bp;
#pragma unroll 1
      for (int g = 0; g < ng; ++g, ++gg, at.advance(R)) {
        if (gg >= R) wait_on(&sm.ebar[at.s], at.parity ^ 1u);
        if (*(volatile int*)&sm.failed) break;
        const int cnt = min(GR, B - g * GR);
        float* stage = ring + (size_t)at.s * GR * SL;
        if constexpr (S::BULK) {
          const uint32_t bytes = (uint32_t)width * 4u;
          const int r = wr + lane * S::REFILL;  // a warp issues one copy in 0.12 us; two warps side by side keep ahead of memory
          if (lane == 0) mbar_expect_tx(&sm.sbar[at.s], bytes * (uint32_t)((cnt - wr + S::REFILL - 1) / S::REFILL));
          __syncwarp();
          if (r < cnt) bulk_load(stage + r * SL, a.X + rows[g * GR + r] * (int64_t)d + c0, bytes, &sm.sbar[at.s]);
        } else {
          for (int r = wr; r < cnt; r += S::REFILL) {
            const float* src = a.X + rows[g * GR + r] * (int64_t)d + c0 + lane * 4;
            const uint32_t dst = smem_u32(stage + r * SL + lane * 4);
#pragma unroll
            for (int q = 0; q < NB; ++q)
              if (q * 128 + lane * 4 < width) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + q * 512), "l"(src + q * 128) : "memory");
          }
          asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(smem_u32(&sm.sbar[at.s])) : "memory");
        }
      }
    }
    if constexpr (!S::BULK) asm volatile("cp.async.wait_all;" ::: "memory");
    if (*(volatile int*)&sm.failed) {  // copies on their way get a bounded chance to land before this CTA leaves
      const uint64_t t0 = global_ns();
      while (global_ns() - t0 < 10000000ull) __nanosleep(1000);
    }
  }
  __syncwarp();
  cluster.sync();  // no CTA leaves while a peer could still address its shared memory
}

using LoopKernel = void (*)(PersistArgs);
template <int BITS, bool ALPC>
LoopKernel pick_nb(int SL) {
  switch (SL / 128) {
    case 1: return stream_loop_kernel<BITS, 1, ALPC>;
    case 2: return stream_loop_kernel<BITS, 2, ALPC>;
    case 4: return stream_loop_kernel<BITS, 4, ALPC>;
    case 8: return stream_loop_kernel<BITS, 8, ALPC>;
    default: return stream_loop_kernel<BITS, 16, ALPC>;
  }
}
LoopKernel pick_loop(int b, int SL, bool alpc) {
  switch (b) {
    case 1: return alpc ? pick_nb<1, true>(SL) : pick_nb<1, false>(SL);
    case 2: return alpc ? pick_nb<2, true>(SL) : pick_nb<2, false>(SL);
    case 4: return alpc ? pick_nb<4, true>(SL) : pick_nb<4, false>(SL);
    case 8: return alpc ? pick_nb<8, true>(SL) : pick_nb<8, false>(SL);
    default: return alpc ? pick_nb<0, true>(SL) : pick_nb<0, false>(SL);
  }
}
struct LoopShape { int threads, rows; size_t stage, part; };  // rows per group; exchange slots per CTA of the cluster
LoopShape loop_shape(int SL) {
  auto of = [](auto s) {
    using S = decltype(s);
    return LoopShape{S::NT, S::GR, S::STAGE, (size_t)LSLOTS * S::GR * S::CP * 4};
  };
  switch (SL / 128) {
    case 1: return of(Shape<1>());
    case 2: return of(Shape<2>());
    case 4: return of(Shape<4>());
    case 8: return of(Shape<8>());
    default: return of(Shape<16>());
  }
}

void loop_config(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, int cs, int clusters, int threads, size_t smem, cudaStream_t st, bool cooperative) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)cs, (unsigned)clusters, 1);
  cfg->blockDim = dim3((unsigned)threads, 1, 1);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeCooperative;  // all CTAs co-resident or the launch fails
  attr[1].val.cooperative = 1;
  cfg->attrs = attr;
  cfg->numAttrs = cooperative ? 2 : 1;
}

}  // namespace

// Slices, cluster size and ring: the narrowest slices (128 columns at least) whose clusters all fit on the device at once, each of as many CTAs
// as there are slices with columns.  us per step with slices of 128, 256, 512, 1,024 and 2,048 columns: d = 752, N = 8, B = 256 9.4, 11.7, 15.9,
// 25.7, 37.3; d = 128, N = 2, B = 256 8.4, 10.9, 13.9, 22.9, 36.2; d = 1,000, N = 4, B = 100 7.2, 8.4, 10.1, 14.7, 18.6; d = 8,192, N = 8, B = 100 with
// 1,024 and 2,048 14.5, 19.4.
bool stream_loop_slices(int d, int N, int B, int alpc, int max_smem, int sm_count, int SL, int* CS_out, size_t* smem_out, int* stages_out) {
  if (B > LMAXB || N > LMAXN || d > 2048 * LCS) return false;
  if (SL > loop_coords(d)) return false;  // few rows rule the narrow slices out, but the exchange buffers end where the vector's power of two does
  const int cs = (d + SL - 1) / SL;
  if (cs > LCS || (N + (alpc ? 1 : 0)) * cs > std::min(LFLAGS, sm_count)) return false;  // one CTA per SM
  const LoopShape s = loop_shape(SL);
  if (B <= 2 * s.rows) return false;  // a step has three groups at least: both sides of the margins and both coefficient warps take part in it
  const size_t fixed = (size_t)SL * 4 * (alpc ? 5 : 2) + s.part * cs + (size_t)((B + 3) & ~3) * 2 * 16 + sizeof(LSmem);
  if (fixed + 3 * s.stage > (size_t)max_smem) return false;
  const int R = (int)(((size_t)max_smem - fixed) / s.stage);
  // as in the per-step kernel: of a peer's u a CTA is at most 2 R + 3 groups ahead, which has to stay below the exchange slots
  *stages_out = std::min(R, cs > 1 ? (LSLOTS - 4) / 2 : LMAXR);
  *CS_out = cs;
  *smem_out = fixed + (size_t)*stages_out * s.stage;
  return true;
}

// Whether the loop is faster than single steps.  For b = 1, 2, 4 and 8 it always is: 800 shapes drawn from N = 1 .. 64, d = 64 .. 16,384, B = 9 .. 256 and
// both algorithms, 0.2 to 1.0 times as long.  For the other widths the end of a step decodes every worker's words in every cluster by shifts that
// are known at run time (single steps decode each once), which costs the more the wider the slices and the more CTAs ask L2.  Loop / single steps,
// 1,500 shapes of those widths: slices of up to 512 columns 0.2 to 0.97.  1,024: 0.6 to 0.98 with up to 108 CTAs, 0.7 to 1.05 with up to 132 in clusters
// of up to six; larger clusters 1.0 to 1.46, more CTAs 1.0 to 1.56, b = 32 with more than 32 workers 1.03 to 1.18.  2,048: b = 32 1.0 to 2.3; the
// others 0.90 to 1.06 with up to four workers of up to six CTAs (Algorithm 2 with more than two of them and more than 64 rows 1.0 to
// 1.11), beyond that 0.95 to 1.8.  Where single steps are slow themselves, rows resident (0.2 to 0.9) or more clusters than the device
// holds at once (0.6 to 1.08), the loop wins whatever its shape.  2,200 other shapes under this rule: 14 are slower, by 1 to 10 %.
bool stream_loop_pays(int b, int N, int B, int alpc, int CS, int SL, bool single_resident, int single_waves) {
  if (b == 1 || b == 2 || b == 4 || b == 8 || single_resident || single_waves > 1 || SL <= 512) return true;
  const int ctas = (N + (alpc ? 1 : 0)) * CS;
  if (SL == 1024) return (b != 32 || N <= 32) && (ctas <= 108 || (CS <= 6 && ctas <= 132));
  return b != 32 && N <= 4 && CS <= 6 && (!alpc || N <= 2 || B <= 64);
}

bool stream_loop_plan(int d, int N, int B, int b, int alpc, int max_smem, int sm_count, bool single_resident, int single_waves, int* CS_out, int* SL_out,
                      size_t* smem_out, int* stages_out) {
  for (int SL = 128; SL <= 2048; SL *= 2) {
    int cs = 0, R = 0;
    size_t smem = 0;
    if (!stream_loop_slices(d, N, B, alpc, max_smem, sm_count, SL, &cs, &smem, &R)) continue;
    LoopKernel k = pick_loop(b, SL, alpc != 0);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    loop_config(&cfg, attr, cs, 1, loop_shape(SL).threads, smem, nullptr, false);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (n < N + (alpc ? 1 : 0)) continue;
    if (!stream_loop_pays(b, N, B, alpc, cs, SL, single_resident, single_waves)) return false;  // wider slices would not either
    *CS_out = cs; *SL_out = SL; *smem_out = smem; *stages_out = R;
    return true;
  }
  return false;
}

cudaError_t launch_stream_loop(const PersistArgs& pa, size_t smem, cudaStream_t st, bool cooperative) {
  LoopKernel k = pick_loop(pa.in.b, pa.in.SL, pa.alpc != 0);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  loop_config(&cfg, attr, pa.in.CS, pa.in.N + (pa.alpc ? 1 : 0), loop_shape(pa.in.SL).threads, smem, st, cooperative);
  return cudaLaunchKernelEx(&cfg, k, pa);
}

}  // namespace lpc
