// Deployment export: argtop_N(phi) per group (the lambda -> 0 limit of the
// Gumbel-top-N sampler, Sec. 4.2.3; the mode of the mask law of Eq. 8), packed
// as bits, with optional pruned weights (kept copied, pruned +0.0).
#include "roi_launch.h"
#include "roi_tiles.cuh"

namespace roi {
namespace {

// One thread per output word (32 elements); groups that straddle two words are
// ranked by both threads, so no atomics are needed and any M <= 32 works.
__global__ void __launch_bounds__(256) roi_export_kernel(const float* __restrict__ phi, int N, int M, int64_t E,
                                                         uint32_t* __restrict__ bits,
                                                         const uint16_t* __restrict__ W,
                                                         uint16_t* __restrict__ Wp) {
  const int64_t nwords = (E + 31) / 32;
  for (int64_t wi = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; wi < nwords;
       wi += int64_t(gridDim.x) * blockDim.x) {
    const int64_t lo = wi * 32;
    const int64_t hi = lo + 32 < E ? lo + 32 : E;
    uint32_t word = 0;
    for (int64_t g = lo / M; g * M < hi; ++g) {
      float k[32];
      for (int l = 0; l < M; ++l) k[l] = phi[g * M + l];
      const uint32_t gb = topn_bits_dyn(k, N, M);
      for (int l = 0; l < M; ++l) {
        const int64_t e = g * M + l;
        if (e >= lo && e < hi && ((gb >> l) & 1u)) word |= 1u << (e - lo);
      }
    }
    bits[wi] = word;
    if (Wp != nullptr) {
      for (int64_t e = lo; e < hi; ++e) Wp[e] = ((word >> (e - lo)) & 1u) ? W[e] : uint16_t(0);
    }
  }
}

// M = 4 and M = 8 on the tile ring of the mask kernels (roi_tiles.cuh): consecutive lanes
// hold consecutive groups, so shared loads and global stores are contiguous.  Bound by
// memory: what the ring is for here is enough bytes in flight.  18944 x 3584, against
// thread-held loads: 2:4 with pruned weights 108.1 -> 82.5 us (6.69 TB/s), bits alone 69.9
// -> 47.0, compressed 84.0 -> 75.2 (6.43 TB/s); 4:8 with pruned weights 93.4 -> 84.5.
enum ExportMode { kBits, kPruned, kCompressed };

constexpr int kThreads = 512;
template <int M, ExportMode MODE>
struct ExportCfg {
  static constexpr int kGroups = 24 / M;                   // groups per thread and tile
  static constexpr int kStages = MODE == kBits ? 3 : 2;    // 147 KB either way
  static constexpr int kTile = kThreads * kGroups * M;
  static constexpr uint32_t kBytes = MODE == kBits ? 4 : 6;  // staged per element
  static constexpr size_t kSmem = tile_smem_bytes<kTile, kStages>(kBytes);
};

struct ExportArgs {
  const float* phi;
  const uint16_t* W;
  uint32_t* bits;    // kBits, kPruned
  uint16_t* Wp;      // kPruned
  uint32_t* values;  // kCompressed: two kept weights a group
  uint32_t* meta;    // kCompressed
  int64_t E;
  int64_t full_tiles;
  int N;
  unsigned int* status;
  bool wait;  // pdl_begin
};

// The deployment mask of one group.
template <int M>
__device__ __forceinline__ uint32_t export_bits(const float* phi, int N) {
  float k[M];
#pragma unroll
  for (int s = 0; s < M / 4; ++s) {
    const float4 v = reinterpret_cast<const float4*>(phi)[s];
    k[4 * s] = v.x, k[4 * s + 1] = v.y, k[4 * s + 2] = v.z, k[4 * s + 3] = v.w;
  }
  if constexpr (M == 4) {
    return topn_bits4(k, N);
  } else {
    return topn_bits<M>(k, N);
  }
}

// One group per lane (all lanes together; inactive ones only take part in the shuffles).
template <int M, ExportMode MODE>
__device__ __forceinline__ void export_group(const float* phi, const uint16_t* W, int64_t e, bool active,
                                             const ExportArgs& a) {
  const int lane = threadIdx.x & 31;
  const uint32_t bits = active ? export_bits<M>(phi, a.N) : 0u;
  uint32_t code = bits;
  if constexpr (MODE == kPruned) {
    if (active) {
#pragma unroll
      for (int s = 0; s < M / 4; ++s)
        reinterpret_cast<uint2*>(a.Wp + e)[s] = keep4(reinterpret_cast<const uint2*>(W)[s], bits >> (4 * s));
    }
  }
  if constexpr (MODE == kCompressed) {
    if (active) {
      // the two set bits of a 2-of-4 mask: lowest i0, then i1
      const uint32_t i0 = __ffs(bits) - 1u;
      const uint32_t i1 = __ffs(bits & (bits - 1u)) - 1u;
      code = i0 | (i1 << 2);
      const uint2 q = *reinterpret_cast<const uint2*>(W);
      // bytes 2 i0, 2 i0 + 1, 2 i1, 2 i1 + 1 of the group's weights
      const uint32_t sel = (2u * i0) | (2u * i0 + 1u) << 4 | (2u * i1) << 8 | (2u * i1 + 1u) << 12;
      a.values[e >> 2] = __byte_perm(q.x, q.y, sel);
    }
  }
  constexpr int kLanesPerWord = 32 / M;
  uint32_t v = code << ((lane % kLanesPerWord) * M);
#pragma unroll
  for (int o = 1; o < kLanesPerWord; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
  if (active && lane % kLanesPerWord == 0) (MODE == kCompressed ? a.meta : a.bits)[e >> 5] = v;
}

template <int M, ExportMode MODE>
__global__ void __launch_bounds__(kThreads, 1) roi_export_tiles_kernel(ExportArgs a) {
  extern __shared__ __align__(128) uint8_t smem[];
  using C = ExportCfg<M, MODE>;
  constexpr int NARR = MODE == kBits ? 1 : 2;
  pdl_begin(a.wait);
  TileSrc<NARR> src;
  src.ptr[0] = reinterpret_cast<const uint8_t*>(a.phi);
  src.esize[0] = 4;
  if constexpr (NARR == 2) {
    src.ptr[1] = reinterpret_cast<const uint8_t*>(a.W);
    src.esize[1] = 2;
  }
  const bool ok = run_tiles<kThreads, C::kTile, C::kStages, NARR>(
      smem, src, a.full_tiles, a.status, [&](const uint8_t* const* stage, int64_t tile, const auto& release) {
        const float* sphi = reinterpret_cast<const float*>(stage[0]);
        const uint16_t* sW = reinterpret_cast<const uint16_t*>(stage[NARR - 1]);
#pragma unroll
        for (int j = 0; j < C::kGroups; ++j) {
          const int g = threadIdx.x + j * kThreads;
          export_group<M, MODE>(sphi + g * M, sW + g * M, tile * C::kTile + g * M, true, a);
        }
        release();
      });
  if (!ok) return;
  // the ragged tail, from global memory, chunks of kThreads groups over all CTAs
  const int64_t t0 = a.full_tiles * C::kTile;
  const int64_t groups = (a.E - t0) / M;
  for (int64_t g0 = tail_rank(a.full_tiles) * kThreads; g0 < groups; g0 += int64_t(gridDim.x) * kThreads) {
    const bool active = g0 + threadIdx.x < groups;
    const int64_t e = t0 + (g0 + (active ? threadIdx.x : 0)) * M;
    export_group<M, MODE>(a.phi + e, NARR == 2 ? a.W + e : nullptr, e, active, a);
  }
}

template <int M, ExportMode MODE>
int launch_tiles(ExportArgs a, cudaStream_t stream) {
  using C = ExportCfg<M, MODE>;
  static_assert(C::kSmem <= 232448, "shared memory per CTA");
  static bool set[64] = {false};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  auto kern = roi_export_tiles_kernel<M, MODE>;
  if (!set[dev]) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::kSmem)) != cudaSuccess) return -1;
    set[dev] = true;
  }
  a.full_tiles = a.E / C::kTile;
  // small tensors as one ragged tail over as many CTAs as it has chunks (the ring costs
  // them more than it gives)
  if (a.full_tiles < sm_count()) a.full_tiles = 0;
  const int64_t want = a.full_tiles + ((a.E - a.full_tiles * C::kTile) / M + kThreads - 1) / kThreads;
  const int64_t cap = sm_count();
  a.wait = lone_pdl(stream);
  return launch_maybe_pdl(kern, int(want < 1 ? 1 : (want < cap ? want : cap)), kThreads, C::kSmem, stream, a.wait, a);
}

int grid_for(int64_t items, int threads) {
  int64_t blocks = (items + threads - 1) / threads;
  const int64_t cap = int64_t(sm_count()) * 8;
  if (blocks > cap) blocks = cap;
  return int(blocks < 1 ? 1 : blocks);
}

}  // namespace

int launch_export_compressed_2of4(const CompressCall& c) {
  ExportArgs a{};
  a.phi = c.phi;
  a.W = c.W;
  a.values = reinterpret_cast<uint32_t*>(c.values);
  a.meta = c.meta;
  a.E = c.E;
  a.N = 2;
  a.status = c.status;
  return launch_tiles<4, kCompressed>(a, c.stream);
}

int launch_export(const ExportCall& c) {
  if (c.M == 4 || c.M == 8) {
    ExportArgs a{};
    a.phi = c.phi;
    a.W = c.W;
    a.bits = c.bits;
    a.Wp = c.Wp;
    a.E = c.E;
    a.N = c.N;
    a.status = c.status;
    if (c.M == 4) return c.Wp != nullptr ? launch_tiles<4, kPruned>(a, c.stream) : launch_tiles<4, kBits>(a, c.stream);
    return c.Wp != nullptr ? launch_tiles<8, kPruned>(a, c.stream) : launch_tiles<8, kBits>(a, c.stream);
  }
  roi_export_kernel<<<grid_for((c.E + 31) / 32, 256), 256, 0, c.stream>>>(c.phi, c.N, c.M, c.E, c.bits, c.W, c.Wp);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

}  // namespace roi
