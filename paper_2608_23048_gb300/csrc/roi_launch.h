// Host-side launch interface between the C ABI (roi_api.cu) and the kernels.
#pragma once

#include <cmath>
#include <cstdint>
#include <cuda_runtime.h>

#include "roi_common.cuh"

namespace roi {

// Every Philox counter (e_base + e) / 4 of a call of E elements is below 2^32
// (its flat element indices stay below 2^34).
inline bool counters_narrow(const NoiseParams& np, int64_t E) {
  const uint64_t lim = uint64_t(1) << 34;
  return np.e_base <= lim && uint64_t(E) <= lim - np.e_base;
}

// The relaxation of a tau != 1 tile kernel (FastGroup, M = 4, 8).  The plain one leaves groups
// beyond its range, ~69 tau in natural-log units of the keys, to a slow routine; WIDE has no
// range and costs more where no group leaves the plain one's:
// - N = 2 takes WIDE always (kAlwaysWide).  Early in the schedule, on logits of unit spread, it
//   costs the 2:4 forward 3 % and the masked linear 5 % on large tensors (18944 x 3584, tau =
//   0.74: 142 -> 147 us, 149 -> 157; the backwards nothing); from tau lambda = 0.046 on, or
//   0.086 at twice that spread, it takes 2 to 34 % less.
// - 4:8 takes it where groups are likely to leave.  The Gumbel noise alone does below tau = 0.2
//   (one 1.5B-shaped block, forward and backward, plain / WIDE: 347 / 343 us at tau = 0.2, 519 /
//   344 at 0.1, 1338 / 344 at 0.06), logits where their spread is a few times 69 tau lambda
//   (8960 x 1536, forward, unit spread: 42.9 / 45.8 us at tau lambda = 0.063, 58.3 / 45.7 at
//   0.046; twice that spread 43.0 / 45.6 at 0.117, 73.3 / 45.9 at 0.086).  The line keeps twice
//   the unit spread on the WIDE side; unit spread pays 7 % between 0.09 and 0.055 for it.
constexpr float kWideTau = 0.2f;
// WIDE holds the weights of a group behind its leader's capped lead at 2^-100 or more where
// they should vanish, and the backward multiplies such a remainder by 1 / tau once a step:
// up to 2^-100 tau^-N of the gradient.  Below 2^-24 (N log2(1 / tau) <= 76: tau >= 4e-12 at
// N = 2, 2e-6 at 4, 0.0014 at 8, 0.037 at 16) that is rounding; at smaller tau (8:16, tau =
// 1e-10: 2e10 where the gradient is 0) the groups go to the log-space routines.
constexpr float kWideBits = 76.0f;
inline bool wide_holds(int N, float tau) { return float(N) * -log2f(tau) <= kWideBits; }
constexpr float kWideTauLambda = 0.09f;
template <int N>
inline bool wide_range(float tau, const NoiseParams& np) {
  return kAlwaysWide<N> || (wide_holds(N, tau) && (tau <= kWideTau || tau < kWideTauLambda * np.inv_lam));
}
// Patterns on the tile kernels.  2:4 and 2:8 have WIDE ones only (tau != 1); where that does
// not hold they go to the any-(N, M) kernels.
inline bool tile_pattern(int N, int M, float tau) {
  return (N == 4 && M == 8) || (N == 2 && (M == 4 || M == 8) && wide_holds(N, tau));
}
// Whether two calls of a batch take the same relaxation (lambda is each item's own).
inline bool same_range(int N, float tau, const NoiseParams& a, const NoiseParams& b) {
  return N != 4 || tau == 1.0f || wide_range<4>(tau, a) == wide_range<4>(tau, b);
}

struct FwdCall {
  const float* phi;
  const uint16_t* W;
  uint16_t* Wm;
  float* soft;      // nullable
  uint32_t* hard;   // nullable
  bool st;          // straight-through: Wm = W where the hard mask is set, +0 elsewhere
  int64_t E;        // rows * cols
  int N, M;
  float tau;
  NoiseParams np;
  unsigned int* status;
  cudaStream_t stream;
};

struct BwdCall {
  const float* phi;
  const uint16_t* W;
  const uint16_t* dWm;
  float* dphi;
  uint16_t* dW;     // nullable
  const uint32_t* hard_in;  // nullable; straight-through: dW = dWm where set, +0 elsewhere
  float* phi_out;   // nullable; fused AdamW: the logits updated in place (== phi)
  float* m;         // AdamW first and second moments (with phi_out)
  float* v;
  AdamW opt;
  int64_t E;
  int N, M;
  float tau;
  NoiseParams np;
  unsigned int* status;
  cudaStream_t stream;
};

struct ExportCall {
  const float* phi;
  uint32_t* bits;
  const uint16_t* W;  // nullable
  uint16_t* Wp;       // nullable
  int64_t E;
  int N, M;
  unsigned int* status;
  cudaStream_t stream;
};

struct CompressCall {
  const float* phi;
  const uint16_t* W;
  uint16_t* values;  // [E / 2]
  uint32_t* meta;    // [E / 32]
  int64_t E;         // multiple of 32
  unsigned int* status;
  cudaStream_t stream;
};

struct LinearCall {
  const uint16_t* X;    // [T, cols] bf16
  const float* phi;     // [rows, cols]
  const uint16_t* W;    // [rows, cols] bf16
  float* Y;             // [T, rows]
  void* workspace;      // nullable: split-K partials and tickets
  size_t workspace_bytes;
  int64_t T, rows, cols;
  int N, M;
  float tau;
  NoiseParams np;
  unsigned int* status;
  cudaStream_t stream;
};

// Each returns the number of kernels launched (>= 0) or -1 after a CUDA error.
int launch_fwd(const FwdCall& c);
int launch_bwd(const BwdCall& c);
// Many independent tensors on one stream: one launch per tensor, or per run of
// small tensors (multi_small), the tile kernels chained by programmatic dependent
// launch so each may start while the previous one drains (stream order is kept:
// each completes after its predecessor).
int launch_fwd_batch(const FwdCall* calls, int count);
int launch_bwd_batch(const BwdCall* calls, int count);
int launch_export(const ExportCall& c);
int launch_export_compressed_2of4(const CompressCall& c);
// Warp-slice kernels for M = 16, 32 (roi_slice.cu).
bool slice_supported(int N, int M);
// (`alone`: no launch is chained behind)
int launch_slice_fwd(const FwdCall& c, bool pdl, bool alone);
int launch_slice_bwd(const BwdCall& c, bool pdl, bool alone);
// A batch's runs of small tensors, one launch each.
int slice_fwd_run(const FwdCall* calls, int count);
int slice_bwd_run(const BwdCall* calls, int count);
int launch_slice_fwd_multi(const FwdCall* calls, int count, bool pdl);
int launch_slice_bwd_multi(const BwdCall* calls, int count, bool pdl);
// Every other (N, M) (roi_any.cu).
int launch_any_fwd(const FwdCall& c);
int launch_any_bwd(const BwdCall& c);
int launch_noise(const NoiseParams& np, int64_t E, uint32_t* words, float* g, cudaStream_t stream);

// Masked linear forward on the tensor cores (roi_linear.cu).
bool linear_supported(int N, int M);
int linear_splits(int64_t T, int64_t rows, int64_t cols);
size_t linear_workspace_bytes(int64_t T, int64_t rows, int64_t cols);
int launch_masked_linear(const LinearCall& c);

// Launches kern<<<grid, threads, smem, stream>>>(args...), with programmatic stream
// serialization allowed when `pdl` (the kernel then may start before the stream's
// previous kernel has finished).  Returns 1, or -1 after a CUDA error.
template <class... KArgs, class... Args>
int launch_maybe_pdl(void (*kern)(KArgs...), int grid, int threads, size_t smem, cudaStream_t stream, bool pdl,
                     const Args&... args) {
  if (!pdl) {
    kern<<<grid, threads, smem, stream>>>(args...);
    return cudaGetLastError() == cudaSuccess ? 1 : -1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...) == cudaSuccess ? 1 : -1;
}

// Whether a launch that follows arbitrary work on `stream` may be made with programmatic
// stream serialization all the same: its kernel then waits for that work itself
// (pdl_begin), and the launch and the CTAs' start hide behind the end of a predecessor that
// lets dependents in (2 us a call in a row of single calls).  Not under stream capture,
// where the predecessor may be no kernel at all.
inline bool lone_pdl(cudaStream_t stream) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(stream, &s) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return s == cudaStreamCaptureStatusNone;
}

// Streaming multiprocessors of the current device (cached).
int sm_count();

// Grid of a tile kernel over one tensor of E elements (`tiles` full tiles, at most `cap`
// CTAs).  `rounds`: a tensor that takes at most so many rounds of one pair of groups a
// thread over the whole GPU is processed that way, as one ragged tail (tiles = 0): the few
// CTAs that its tiles would occupy, each with a ring to fill, take longer (2:4 at tau = 1,
// forward / backward of 32768 elements 5.3 / 4.5 -> 3.1 / 3.1 us, 896 x 896 5.4 / 4.6 ->
// 4.7 / 4.5).  Launches that are chained behind others (rounds = 0) keep the tiles.
inline int tile_grid(int64_t& tiles, int64_t E, int M, int chunk, int64_t tile, int64_t cap, int rounds) {
  if ((E / M + chunk - 1) / chunk <= rounds * cap) tiles = 0;
  const int64_t chunks = ((E - tiles * tile) / M + chunk - 1) / chunk;
  const int64_t want = tiles + chunks;
  return int(want < 1 ? 1 : (want < cap ? want : cap));
}

// Batched calls: a run of consecutive items with the same tile kernel, each of
// them small (fewer than kMultiTilesPerSm full tiles per SM), goes to one
// multi-tensor launch when it holds at least multi_min_run items.  One launch per
// small tensor spends much of its time on fixed costs (ring fill and drain, the
// ragged tail, the gap to the next launch).  A larger tensor keeps a launch of its
// own: the multi-tensor kernels hold the current tensor's arguments in registers
// rather than in the constant bank, and measured 4-7 % slower on 18944 x 3584
// tensors.  That per-tile cost also decides the run lengths: the plain backward
// gains from runs of 2 (the q, k, v, o tensors of a 7B-shaped layer), while the
// forward and the backward fused with AdamW lost on those runs (7B-shaped 2:4 step,
// forward 11.72 -> 11.80 ms, fused backward 28.8 -> 29.0 ms) and gain only over long
// ones.  A fwd + bwd step over a
// Qwen2.5-shaped layer set went from 1.90 to 1.57 ms (0.5B-shaped, 2:4: one launch
// per direction), 8.92 to 8.78 ms (1.5B-shaped, 4:8) and 24.31 to 24.19 ms
// (7B-shaped, 2:4).
constexpr int64_t kMultiTilesPerSm = 12;
inline int multi_min_run(bool short_runs_pay) { return short_runs_pay ? 2 : 8; }
inline bool multi_small(int64_t E, int64_t tile) { return E / tile < kMultiTilesPerSm * sm_count(); }

}  // namespace roi
