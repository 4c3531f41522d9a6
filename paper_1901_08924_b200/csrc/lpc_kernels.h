// Internal launch interface between the C ABI (lpc_api.cu) and the kernel files.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "lpc_scale.h"

namespace lpc {

constexpr int TILE = 8192;  // coordinates per CTA tile of the standalone quantizer / aggregator kernels

// Launches a kernel that calls wait_for_launch_before, so that it overlaps with the tail of the kernel before it.
template <class... Params, class... Args>
cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// One tensor segment of a (segmented) vector.
struct SegInfo {
  int64_t off;         // first element in the vector
  int64_t len;         // elements
  int64_t word_off;    // first word of its packed stream inside a worker's stream (multiple of 4)
  int64_t pad_words;   // words reserved for it (multiple of 4)
  uint32_t block_base; // first Philox block of its rounding stream
  int32_t tile_first;  // first tile index
  int32_t tile_count;
  int32_t pad_;
};

struct ScaleRec {  // result of the scale rule for one (worker, segment)
  float delta, rdelta, T, lower;
  uint32_t flags, pad0, pad1, pad2;  // flags: bit 0 degenerate, bit 1 non-finite input, SCALE_NONE_OUTSIDE
};
constexpr uint32_t SCALE_NONE_OUTSIDE = 4u;  // the threshold is the largest magnitude: no coordinate is outside the hull

struct QuantArgs {
  const float* U;
  const float* U_sub;  // nullable
  int64_t ld;
  int N;
  int b;
  int clip_mode;
  float clip_value;
  uint64_t seed;
  uint64_t k;
  const SegInfo* segs;     // device, nseg entries
  const int32_t* tile_seg; // device, ntiles entries
  int nseg;
  int ntiles;
  // scratch
  uint32_t* pmax;  // N * ntiles
  float* ps1;      // N * ntiles
  float* ps2;      // N * ntiles
  ScaleRec* scales;  // N * nseg
  // outputs
  uint32_t* codes;
  int64_t stride_words;
  float* delta_out;       // N * nseg
  uint32_t* clipped_out;  // N * nseg, cleared with the scale (never null: internal scratch when the caller gives none)
  int count_clipped;      // 0: skip counting the coordinates outside the hull (the counts stay zero)
  int shared_scale;       // 1: every worker quantizes with delta_t = max_i delta_t^i (schemes (b), (c) of Section 3.2)
  unsigned int* dev_status;
};

// hook(user, kind, begin) is called around each kernel of the sequence (kind = LPC_KERNEL_* of lpc.h) when non-null.
typedef void (*LaunchHook)(void* user, int kind, int begin);
// Tiles per CTA of the second pass, and whether the run of tiles that starts at tile0 consists of whole tiles of one
// segment (the condition, besides 16-byte aligned vectors and a non-degenerate scale, for its pipelined loop).
int quantize_run_tiles();
int quantize_pack_launches(const QuantArgs& a);  // kernels that launch_quantize_pack launches
cudaError_t launch_quantize_pack(const QuantArgs& a, int kept_tiles, int sm_count, cudaStream_t st, LaunchHook hook = nullptr, void* user = nullptr);
// The same for short vectors, one cluster per worker and nothing looked at twice.
// Tiles at the end that the first look leaves in L2 for the second (0: no cache policy).  offsets_aligned says that every segment's offset is a multiple of 8; l2_bytes is the size of the device's L2.
int quantize_kept_tiles(const QuantArgs& a, bool offsets_aligned, int64_t l2_bytes);
bool quantize_fits_cluster(const QuantArgs& a, int sm_count);
cudaError_t launch_quantize_cluster(const QuantArgs& a, cudaStream_t st);

// One look at the values for many messages with a subtrahend (lpc_quantize_once.cu).
struct QuantOnceArgs {
  QuantArgs q;                // pmax, ps1, ps2 and scales are not used
  ulonglong2* partials;       // one per tile of every worker, zero before the first call: max |u|, S1, S2 and the call's tag
  unsigned long long* counts; // N * nseg, zero between calls (also after one whose waits ran out)
  unsigned int* epoch;        // the call's tag: 1 before the first call, moved on by each
  unsigned int* done;         // zero between calls
  float levels, inv_levels;   // as in ScaleRule
  int stop_at;                // -1; else CTA 0 goes no further than this many tiles, as after a wait that ran out
};
// Whether a call takes that path.  max_tiles: tiles of the longest message; offsets_x4: every segment's offset is a multiple of 4.
bool quantize_takes_one_look(const QuantArgs& a, int64_t len, int max_tiles, bool offsets_x4, int sm_count, int64_t l2_bytes);
cudaError_t launch_quantize_once(const QuantOnceArgs& oa, int sm_count, cudaStream_t st);

struct AggArgs {
  const uint32_t* codes;
  int64_t stride_words;
  const float* delta;  // N * nseg
  int N;
  int b;
  int divisor;      // the decoded sum is divided by this count: N for Eq. 3; the worker count behind a server's sum stream
  const SegInfo* segs;
  const int32_t* tile_seg;
  int nseg;
  int ntiles;
  const float* mu;  // nullable
  float* x;         // in/out
  float eta;
  float lambda_l1;
  float* v_out;     // nullable
  uint64_t* k_counter;  // nullable: incremented by k_step when the kernel finishes (graph replay)
  uint64_t k_step;
  // mode 1 (Algorithm 2, steps 12-13): x is read only (the coupled point x_{k+1}) and instead of the
  // proximal step on x the kernel updates  y = soft(x - inv4L*v, inv4L*lambda_l1),
  // z = soft(z - alpha*vhat, alpha*lambda_l1),  ysum += y.
  int mode;
  float* y;
  float* z;
  float* ysum;
  const float* vhat;
  float alpha;
  float inv4L;
  // strongly convex case of Algorithm 2, h = lambda_l1*||.||_1 + (sigma/2)*||.||^2: the soft-threshold results are
  // multiplied by cy = 1/(1 + sigma*inv4L) and cz = 1/(1 + alpha*sigma), and ysum += wy * y (the snapshot weight
  // (1 + alpha*sigma)^t of the step).  All three are 1 in the general convex case, where they change no bit.
  float cy, cz, wy;
  int split;  // CTAs per tile (1, 2 or 4): aggregate_split(ntiles, sm_count), set by the caller
};

// CTAs that share one tile of the aggregator: below two waves of resident CTAs (4 per SM) a tile's sweeps are spread
// over 2 or 4 CTAs so that short vectors still fill the machine.
int aggregate_split(int ntiles, int sm_count);
cudaError_t launch_unpack_average_prox(const AggArgs& a, cudaStream_t st);

// The server of the parameter-server schemes (Section 3.2): N code streams of b bits on one grid in, one stream out.
struct ServerArgs {
  const uint32_t* codes;   // N streams, stream i at codes + i * stride_words, segment layout `segs`
  int64_t stride_words;
  int N;
  int b;
  int b_out;               // scheme (b): b + ceil(log2 N), index sums; scheme (c): b, re-quantized average
  int requantize;
  uint64_t seed;
  uint64_t k;
  const SegInfo* segs;     // layout of the input streams (width b)
  const SegInfo* segs_out; // layout of the output stream (width b_out): same segments and tiles, other word offsets
  const int32_t* tile_seg;
  int nseg;
  int ntiles;
  uint32_t* out;
};
cudaError_t launch_server_reduce(const ServerArgs& a, cudaStream_t st);

// Histogram of the code values of every (worker, segment) message: hist[(worker * nseg + seg) * 2^b + code].
struct HistArgs {
  const uint32_t* codes;
  int64_t stride_words;
  int N;
  int b;                   // 1..8
  const SegInfo* segs;
  const int32_t* tile_seg;
  int nseg;
  int ntiles;
  unsigned long long* hist;  // N * nseg * 2^b counts, added to (the caller clears them)
};
cudaError_t launch_code_histogram(const HistArgs& a, int sm_count, cudaStream_t st);
// Entropy bound and Huffman length of `messages` histograms of 2^b counts each; the outputs may be pinned host memory.
cudaError_t launch_coded_size(const unsigned long long* hist, int messages, int b, double* entropy_out,
                              unsigned long long* huffman_out, cudaStream_t st);

}  // namespace lpc

namespace lpc {
cudaError_t launch_loop_scales(const uint32_t* max_bits, const float* S1, const float* S2, int64_t count, const ScaleRule& rule, int b,
                               int clip_mode, float clip_value, float4* scale_out, uint32_t* flags_out, cudaStream_t st);
cudaError_t launch_stream_blocks(uint64_t seed, uint32_t tag, uint32_t worker, uint64_t k, uint32_t block0,
                                 int64_t count, uint32_t* out, cudaStream_t st);
}  // namespace lpc
