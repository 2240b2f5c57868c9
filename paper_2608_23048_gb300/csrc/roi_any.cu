// Any 1 <= N < M <= 32 without a kernel of its own (1:4, 3:4, 1:2, 3:7, 4:16, ...): the same
// method as the tile kernels (Sec. 4.2.2 Eq. 10-12, Algorithm 1; Eq. 5; backward through
// the relaxation) with N and M at run time.  A thread holds whole groups, padded to MP = 4,
// 8, 16 or 32 members whose keys lie far below every real one: two groups in lockstep on
// packed FP32 for MP <= 8, one for the wider ones.  The relaxation is FastGroup's WIDE one
// (finite keys never leave its range) with the step loop rolled, and the backward keeps
// the steps' weights in thread-local memory.  Non-finite keys go to ExactGroup in place; at a
// tau too small for WIDE (wide_holds) all groups go to kernels of ExactGroup alone.
#include "roi_launch.h"

namespace roi {
namespace {

constexpr int kThreads = 128;
// CTAs per SM that the register budget is sized for: the padded group without a spill, and no
// more registers than that (left to itself ptxas spills at MP = 4, forward and backward, and in
// the backward at 8: 3:4 at 1536 x 1536 backward 15.8 us, 12.2 here; with 6 CTAs at MP = 4 the
// forward takes 11.5 us, with 8 11.2).
template <int MP>
constexpr int kMinBlocks = MP == 4 ? 8 : MP <= 16 ? 4 : 2;
// Padding members' keys (log2 units), the magnitude (squared) up to which real keys take the fast
// relaxation, and the padding's largest offset from the second largest key over tau: 2^x is 0
// there whatever tau is, and second_of never picks it (a real key's offset lies above the
// padding's by 2e18 / tau and by 1e30 - 2e18 / tau, of which one is 5e29 or more).
constexpr float kPadKey = -3.0e18f;
constexpr float kMaxKeySq = 1.0e36f;
constexpr float kPadOffset = -1.0e30f;

struct AnyArgs {
  const float* phi;
  const uint16_t* W;
  const uint16_t* dWm;
  uint16_t* Wm;
  float* soft;              // nullable
  uint32_t* hard;           // nullable
  bool st;                  // straight-through forward
  float* dphi;              // nullable with phi_out
  uint16_t* dW;             // nullable
  const uint32_t* hard_in;  // nullable
  float* phi_out;           // nullable: fused AdamW
  float* m;
  float* v;
  AdamW opt;
  int64_t groups;
  int N, M;
  float tau, inv_tau;
  NoiseParams np;
  bool wait;  // pdl_begin
};

template <int MP>
struct Lanes {
  using V = F2;
};
template <>
struct Lanes<16> {
  using V = float;
};
template <>
struct Lanes<32> {
  using V = float;
};

template <class V>
__device__ __forceinline__ float lane_of(V v, int h) {
  if constexpr (vlanes<V>() == 1) {
    return v;
  } else {
    return h == 0 ? lo(v) : hi(v);
  }
}
template <class V>
__device__ __forceinline__ V from_lanes(const float (&x)[vlanes<V>()]) {
  if constexpr (vlanes<V>() == 1) {
    return x[0];
  } else {
    return f2(x[0], x[1]);
  }
}

// One bf16 member each of groups e0[h], l < M; 0 beyond.
template <int MP, class V>
__device__ __forceinline__ void load_bf16(const uint16_t* p, const int64_t* e0, int M, V (&out)[MP]) {
  constexpr int L = vlanes<V>();
#pragma unroll
  for (int s = 0; s < MP / 4; ++s) {
    float x[4][L];
#pragma unroll
    for (int h = 0; h < L; ++h) {
      if ((M & 3) == 0) {
        const uint2 q = 4 * s < M ? *reinterpret_cast<const uint2*>(p + e0[h] + 4 * s) : make_uint2(0u, 0u);
        x[0][h] = bf16_bits_to_float(q.x & 0xffffu), x[1][h] = bf16_bits_to_float(q.x >> 16);
        x[2][h] = bf16_bits_to_float(q.y & 0xffffu), x[3][h] = bf16_bits_to_float(q.y >> 16);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) x[j][h] = 4 * s + j < M ? bf16_bits_to_float(p[e0[h] + 4 * s + j]) : 0.0f;
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) out[4 * s + j] = from_lanes<V>(x[j]);
  }
}

// Keys in log2 units of the groups at e0[h] (call-flat first elements), padding beyond M.
template <int MP, class V>
__device__ __forceinline__ void any_keys(const AnyArgs& a, const int64_t* e0, V (&kap)[MP]) {
  constexpr int L = vlanes<V>();
  uint4 block[L] = {};
#pragma unroll
  for (int s = 0; s < MP / 4; ++s) {
    float ph[4][L], one_plus[4][L];
#pragma unroll
    for (int h = 0; h < L; ++h) {
      const uint64_t e = a.np.e_base + uint64_t(e0[h]) + 4 * s;
      if ((a.M & 3) == 0) {  // groups start on a noise block then
        if (4 * s < a.M) {
          const float4 p = *reinterpret_cast<const float4*>(a.phi + e0[h] + 4 * s);
          const uint4 x = noise_block(a.np, e);
          ph[0][h] = p.x, ph[1][h] = p.y, ph[2][h] = p.z, ph[3][h] = p.w;
          one_plus[0][h] = one_plus_from_word(x.x), one_plus[1][h] = one_plus_from_word(x.y);
          one_plus[2][h] = one_plus_from_word(x.z), one_plus[3][h] = one_plus_from_word(x.w);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) ph[j][h] = 0.0f, one_plus[j][h] = 1.5f;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          ph[j][h] = 0.0f, one_plus[j][h] = 1.5f;
          if (4 * s + j < a.M) {
            ph[j][h] = a.phi[e0[h] + 4 * s + j];
            const uint32_t w = uint32_t(e + j) & 3u;
            if (w == 0u || 4 * s + j == 0) block[h] = noise_block(a.np, (e + j) & ~uint64_t(3));
            one_plus[j][h] = one_plus_from_word(w == 0u ? block[h].x : w == 1u ? block[h].y : w == 2u ? block[h].z : block[h].w);
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      // u = (1 + k 2^-23) - (1 - 2^-24), exact (see uniform_from_word)
      const V u = vsub(from_lanes<V>(one_plus[j]), vconst<V>(__uint_as_float(0x3f7fffffu)));
      const V k = key_log2(from_lanes<V>(ph[j]), u, a.np.l2e_inv_lam);
      kap[4 * s + j] = 4 * s + j < a.M ? k : vconst<V>(kPadKey);
    }
  }
}

// The keys of one group for ExactGroup, in natural-log units: phi / lambda stays finite up to the
// type's largest value, where log2 units overflow (the lowest one masks a member out).
__device__ __forceinline__ void exact_keys(const AnyArgs& a, int64_t e0, float* kap) {
  uint4 block = {};
  for (int l = 0; l < a.M; ++l) {
    const uint64_t e = a.np.e_base + uint64_t(e0) + l;
    const uint32_t w = uint32_t(e) & 3u;
    if (w == 0u || l == 0) block = noise_block(a.np, e & ~uint64_t(3));
    kap[l] = __fmaf_rn(a.phi[e0 + l], a.np.inv_lam,
                       gumbel_from_word(w == 0u ? block.x : w == 1u ? block.y : w == 2u ? block.z : block.w));
  }
}

// Sum over the other members, of which the padding's are 0.
template <int MP, class V>
__device__ __forceinline__ void others_of(const V (&x)[MP], V (&ex)[MP]) {
  if constexpr (MP <= 8) {
    exclusive_sums(x, ex);
  } else {
    exclusive_sums_scalar(x, ex);
  }
}
template <int MP, class V>
__device__ __forceinline__ V total_of(const V (&x)[MP]) {
  V t[MP];
#pragma unroll
  for (int l = 0; l < MP; ++l) t[l] = x[l];
#pragma unroll
  for (int w = MP / 2; w >= 1; w >>= 1)
#pragma unroll
    for (int l = 0; l < w; ++l) t[l] = vadd(t[l], t[l + w]);
  return t[0];
}

// FastGroup's WIDE forward with N steps at run time; step(k, mu) sees every step's weights.
// Returns the lanes' flags (a non-finite key, or keys beyond kMaxKeySq).
template <int MP, class V, class Step>
__device__ __forceinline__ uint32_t any_relax(const V (&kap)[MP], int N, int M, float inv_tau, Step&& step) {
  const V itau = vconst<V>(inv_tau);
  V sq = vmul(kap[0], kap[0]);
#pragma unroll
  for (int l = 1; l < MP; ++l)
    if (l < M) sq = vfma(kap[l], kap[l], sq);
  const uint32_t flag = vbelow(vsub(vconst<V>(kMaxKeySq), sq), 0.0f);
  V x[MP];
  V ref = second_of(kap);
#pragma unroll
  for (int l = 0; l < MP; ++l) {
    x[l] = vmul(vsub(kap[l], ref), itau);
    if (l >= MP / 2 && l >= M) x[l] = vmin(x[l], vconst<V>(kPadOffset));
  }
#pragma unroll 1
  for (int k = 0; k < N; ++k) {
    V c[MP], e[MP];
#pragma unroll
    for (int l = 0; l < MP; ++l) {
      c[l] = vmin(x[l], vconst<V>(kLeadCap));
      e[l] = vmap(c[l], ex2_approx);
    }
    const V r = vmap(total_of(e), rcp_approx);
    V mu[MP];
#pragma unroll
    for (int l = 0; l < MP; ++l) mu[l] = vmul(e[l], r);
    step(k, mu);
    if (k + 1 < N) {
      V ex[MP];
      others_of(e, ex);
#pragma unroll
      for (int l = 0; l < MP; ++l)
        x[l] = vfma(vsub(vmap(vmul(ex[l], r), lg2_approx), vsub(x[l], c[l])), itau, x[l]);
      ref = second_of(x);
#pragma unroll
      for (int l = 0; l < MP; ++l) x[l] = vsub(x[l], ref);
    }
  }
  return flag;
}

// The first elements of this thread's groups (groups L t + h; the last thread's second
// group may not exist and then doubles its first) and how many exist.
template <int L>
__device__ __forceinline__ int any_groups(const AnyArgs& a, int64_t t, int64_t (&e0)[L]) {
  const int64_t g = t * L;
  const int have = g + L <= a.groups ? L : (g < a.groups ? int(a.groups - g) : 0);
#pragma unroll
  for (int h = 0; h < L; ++h) e0[h] = (have == 0 ? 0 : h < have ? g + h : g) * a.M;
  return have;
}

template <int MP>
__global__ void __launch_bounds__(kThreads, kMinBlocks<MP>) roi_any_fwd_kernel(AnyArgs a, bool words) {
  using V = typename Lanes<MP>::V;
  constexpr int L = vlanes<V>();
  pdl_begin(a.wait);
  const int64_t lanes = (a.groups + L - 1) / L;
  const int64_t stride = int64_t(gridDim.x) * kThreads;
  for (int64_t t0 = int64_t(blockIdx.x) * kThreads; t0 < lanes; t0 += stride) {
    int64_t e0[L];
    const int have = any_groups<L>(a, t0 + threadIdx.x, e0);
    uint32_t bits[L] = {};
    if (have > 0) {
      V kap[MP], S[MP];
      any_keys<MP, V>(a, e0, kap);
#pragma unroll
      for (int l = 0; l < MP; ++l) S[l] = vconst<V>(0.0f);
      const uint32_t flag = any_relax<MP, V>(kap, a.N, a.M, a.inv_tau, [&](int, const V (&mu)[MP]) {
#pragma unroll
        for (int l = 0; l < MP; ++l) S[l] = vadd(S[l], mu[l]);
      });
      V w[MP];
      load_bf16<MP, V>(a.W, e0, a.M, w);
#pragma unroll
      for (int h = 0; h < L; ++h) {
        if (h >= have) break;
        float s[MP], k[MP];
#pragma unroll
        for (int l = 0; l < MP; ++l) s[l] = lane_of(S[l], h), k[l] = lane_of(kap[l], h);
        const bool rank = a.hard != nullptr || a.st;
        if ((flag >> h) & 1u) {
          float kn[MP];
          exact_keys(a, e0[h], kn);
          ExactGroup<MP - 1, MP> ex;
          ex.forward(kn, a.N, a.M, a.tau, s);
          if (rank) bits[h] = topn_bits_dyn(kn, a.N, a.M);
        } else if (rank) {
          if constexpr (MP == 4) {
            bits[h] = topn_bits4(k, a.N);
          } else {
            bits[h] = topn_bits<MP>(k, a.N);
          }
        }
        if ((a.M & 3) == 0) {
#pragma unroll
          for (int q = 0; q < MP / 4; ++q) {
            if (4 * q < a.M) {
              const int64_t e = e0[h] + 4 * q;
              uint2 o;
              if (a.st) {
                o = keep4(*reinterpret_cast<const uint2*>(a.W + e), bits[h] >> (4 * q));
              } else {
                o.x = pack_bf16x2(__fmul_rn(lane_of(w[4 * q], h), s[4 * q]), __fmul_rn(lane_of(w[4 * q + 1], h), s[4 * q + 1]));
                o.y = pack_bf16x2(__fmul_rn(lane_of(w[4 * q + 2], h), s[4 * q + 2]),
                                  __fmul_rn(lane_of(w[4 * q + 3], h), s[4 * q + 3]));
              }
              *reinterpret_cast<uint2*>(a.Wm + e) = o;
              if (a.soft != nullptr)
                *reinterpret_cast<float4*>(a.soft + e) = make_float4(s[4 * q], s[4 * q + 1], s[4 * q + 2], s[4 * q + 3]);
            }
          }
        } else {
#pragma unroll
          for (int l = 0; l < MP; ++l) {
            if (l < a.M) {
              const int64_t e = e0[h] + l;
              a.Wm[e] = a.st ? (((bits[h] >> l) & 1u) ? a.W[e] : uint16_t(0))
                             : __bfloat16_as_ushort(__float2bfloat16_rn(__fmul_rn(lane_of(w[l], h), s[l])));
              if (a.soft != nullptr) a.soft[e] = s[l];
            }
          }
        }
      }
    }
    if (a.hard != nullptr) {
      if (words) {
        // M divides 32: 32 / (L M) consecutive lanes fill a word
        const int per = 32 / (L * a.M) > 0 ? 32 / (L * a.M) : 1;
        uint32_t v = bits[0];
        if constexpr (L == 2) v |= bits[1] << a.M;
        v <<= (int(threadIdx.x) & (per - 1)) * L * a.M;
        for (int o = 1; o < per; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
        if (have > 0 && (int(threadIdx.x) & (per - 1)) == 0) a.hard[e0[0] >> 5] = v;
      } else {
#pragma unroll
        for (int h = 0; h < L; ++h) {
          if (h < have) {
            const uint64_t v = uint64_t(bits[h]) << (e0[h] & 31);
            if (uint32_t(v) != 0u) atomicOr(&a.hard[e0[h] >> 5], uint32_t(v));
            if (uint32_t(v >> 32) != 0u) atomicOr(&a.hard[(e0[h] >> 5) + 1], uint32_t(v >> 32));
          }
        }
      }
    }
  }
}

template <int MP>
__global__ void __launch_bounds__(kThreads, kMinBlocks<MP>) roi_any_bwd_kernel(AnyArgs a) {
  using V = typename Lanes<MP>::V;
  constexpr int L = vlanes<V>();
  pdl_begin(a.wait);
  const V itau = vconst<V>(a.inv_tau);
  const int64_t lanes = (a.groups + L - 1) / L;
  const int64_t stride = int64_t(gridDim.x) * kThreads;
  for (int64_t t = int64_t(blockIdx.x) * kThreads + threadIdx.x; t < lanes; t += stride) {
    int64_t e0[L];
    const int have = any_groups<L>(a, t, e0);
    // mu of every step; ExactGroup, which comes after the sweep, keeps its own in the same place
    union {
      V mu[MP - 1][MP];
      ExactGroup<MP - 1, MP> exact;
    } steps;
    V(&hist)[MP - 1][MP] = steps.mu;
    V kap[MP], c[MP], b[MP];
    any_keys<MP, V>(a, e0, kap);
    const uint32_t flag = any_relax<MP, V>(kap, a.N, a.M, a.inv_tau, [&](int k, const V (&mu)[MP]) {
#pragma unroll
      for (int l = 0; l < MP; ++l) hist[k][l] = mu[l];
    });
    {
      V w[MP];
      load_bf16<MP, V>(a.W, e0, a.M, w);
      load_bf16<MP, V>(a.dWm, e0, a.M, c);
#pragma unroll
      for (int l = 0; l < MP; ++l) c[l] = vmul(c[l], w[l]);
    }
    // FastGroup's sweep with b = tau dL/dkappa
    {
      V cm[MP];
#pragma unroll
      for (int l = 0; l < MP; ++l) cm[l] = vmul(c[l], hist[a.N - 1][l]);
      const V cmu = total_of(cm);
#pragma unroll
      for (int l = 0; l < MP; ++l) b[l] = vmul(hist[a.N - 1][l], vsub(c[l], cmu));
    }
#pragma unroll 1
    for (int k = a.N - 2; k >= 0; --k) {
      V mk[MP], t1[MP], t2[MP];
#pragma unroll
      for (int l = 0; l < MP; ++l) mk[l] = hist[k][l];
#pragma unroll
      for (int l = 0; l < MP; ++l) t1[l] = vfma(b[l], itau, vmul(c[l], mk[l]));
      const V K = total_of(t1);
      others_of(mk, t1);  // 1 - mu
#pragma unroll
      for (int l = 0; l < MP; ++l) t1[l] = vmul(b[l], vmap(t1[l], rcp_approx));
      others_of(t1, t2);
#pragma unroll
      for (int l = 0; l < MP; ++l) b[l] = vfma(mk[l], vfma(t2[l], itau, vsub(c[l], K)), b[l]);
    }
    V S[MP];
#pragma unroll
    for (int l = 0; l < MP; ++l) S[l] = vconst<V>(0.0f);
    if (a.dW != nullptr && a.hard_in == nullptr) {
#pragma unroll 1
      for (int k = 0; k < a.N; ++k)
#pragma unroll
        for (int l = 0; l < MP; ++l) S[l] = vadd(S[l], hist[k][l]);
    }
    const V scale = vconst<V>(a.inv_tau * a.np.inv_lam);
#pragma unroll
    for (int l = 0; l < MP; ++l) b[l] = vmul(b[l], scale);
#pragma unroll
    for (int h = 0; h < L; ++h) {
      if (h >= have) break;
      float g[MP], s[MP];
#pragma unroll
      for (int l = 0; l < MP; ++l) g[l] = lane_of(b[l], h), s[l] = lane_of(S[l], h);
      if ((flag >> h) & 1u) {
        float kn[MP], cc[MP];
#pragma unroll
        for (int l = 0; l < MP; ++l) cc[l] = lane_of(c[l], h);
        exact_keys(a, e0[h], kn);
        steps.exact.forward(kn, a.N, a.M, a.tau, s);
        steps.exact.backward(cc, a.N, a.M, a.tau, g);
#pragma unroll
        for (int l = 0; l < MP; ++l) g[l] *= a.np.inv_lam;
      }
#pragma unroll
      for (int q = 0; q < MP / 4; ++q) {
        if (4 * q >= a.M) break;
        const int64_t e = e0[h] + 4 * q;
        if ((a.M & 3) == 0) {
          const float g4[4] = {g[4 * q], g[4 * q + 1], g[4 * q + 2], g[4 * q + 3]};
          if (a.dphi != nullptr) *reinterpret_cast<float4*>(a.dphi + e) = make_float4(g4[0], g4[1], g4[2], g4[3]);
          if (a.phi_out != nullptr)
            adamw4(a.phi_out, a.m, a.v, e, *reinterpret_cast<const float4*>(a.phi + e), g4, a.opt);
          if (a.dW != nullptr) {
            const uint2 d = *reinterpret_cast<const uint2*>(a.dWm + e);
            uint2 o;
            if (a.hard_in != nullptr) {
              o = keep4(d, hard4(a.hard_in, e));
            } else {
              o.x = pack_bf16x2(__fmul_rn(bf16_bits_to_float(d.x & 0xffffu), s[4 * q]),
                                __fmul_rn(bf16_bits_to_float(d.x >> 16), s[4 * q + 1]));
              o.y = pack_bf16x2(__fmul_rn(bf16_bits_to_float(d.y & 0xffffu), s[4 * q + 2]),
                                __fmul_rn(bf16_bits_to_float(d.y >> 16), s[4 * q + 3]));
            }
            *reinterpret_cast<uint2*>(a.dW + e) = o;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (4 * q + j >= a.M) break;
            const int64_t el = e + j;
            if (a.dphi != nullptr) a.dphi[el] = g[4 * q + j];
            if (a.phi_out != nullptr) {
              float ph = a.phi[el], mm = a.m[el], vv = a.v[el];
              adamw_elem(ph, g[4 * q + j], mm, vv, a.opt);
              a.phi_out[el] = ph;
              a.m[el] = mm;
              a.v[el] = vv;
            }
            if (a.dW != nullptr) {
              if (a.hard_in != nullptr) {
                a.dW[el] = ((a.hard_in[el >> 5] >> (el & 31)) & 1u) ? a.dWm[el] : uint16_t(0);
              } else {
                a.dW[el] = __bfloat16_as_ushort(__float2bfloat16_rn(__fmul_rn(bf16_bits_to_float(a.dWm[el]), s[4 * q + j])));
              }
            }
          }
        }
      }
    }
  }
}

// Every group by ExactGroup, one a thread, members in local memory (1536 x 1536, tau = 0.05,
// forward / backward: 18:24 1341 / 3828 us in place behind a fast relaxation that was thrown
// away, 941 / 2529 here; 20:32 1531 / 4906, 1297 / 4070).  What bounds these is the L1's
// bandwidth for the members.  A warp's frame is 32 times a thread's: the keys' array is longer
// than 32 so that the frame is 16 bytes times an odd number and the warps' frames start in
// different sets of the L1 (20:32 with 4864 B a thread 1516 / 4887 us, with 4880 1297 / 4070).
constexpr int kExactKeys = 36;
// hard words are zeroed beforehand
__global__ void __launch_bounds__(kThreads) roi_any_exact_fwd_kernel(AnyArgs a) {
  pdl_begin(a.wait);
  const int64_t stride = int64_t(gridDim.x) * kThreads;
  for (int64_t g = int64_t(blockIdx.x) * kThreads + threadIdx.x; g < a.groups; g += stride) {
    const int64_t e0 = g * a.M;
    float kap[kExactKeys], S[32];
    exact_keys(a, e0, kap);
    const uint32_t bits = a.hard != nullptr || a.st ? topn_bits_dyn(kap, a.N, a.M) : 0u;
    ExactGroup<31, 32> ex;
    ex.forward(kap, a.N, a.M, a.tau, S);
    for (int l = 0; l < a.M; ++l) {
      const int64_t e = e0 + l;
      a.Wm[e] = a.st ? (((bits >> l) & 1u) ? a.W[e] : uint16_t(0))
                     : __bfloat16_as_ushort(__float2bfloat16_rn(__fmul_rn(bf16_bits_to_float(a.W[e]), S[l])));
      if (a.soft != nullptr) a.soft[e] = S[l];
    }
    if (a.hard != nullptr) {
      const uint64_t v = uint64_t(bits) << (e0 & 31);
      if (uint32_t(v) != 0u) atomicOr(&a.hard[e0 >> 5], uint32_t(v));
      if (uint32_t(v >> 32) != 0u) atomicOr(&a.hard[(e0 >> 5) + 1], uint32_t(v >> 32));
    }
  }
}

__global__ void __launch_bounds__(kThreads) roi_any_exact_bwd_kernel(AnyArgs a) {
  pdl_begin(a.wait);
  const int64_t stride = int64_t(gridDim.x) * kThreads;
  for (int64_t g = int64_t(blockIdx.x) * kThreads + threadIdx.x; g < a.groups; g += stride) {
    const int64_t e0 = g * a.M;
    float kap[kExactKeys], c[32], S[32], dk[32];
    exact_keys(a, e0, kap);
    for (int l = 0; l < a.M; ++l) c[l] = __fmul_rn(bf16_bits_to_float(a.dWm[e0 + l]), bf16_bits_to_float(a.W[e0 + l]));
    ExactGroup<31, 32> ex;
    ex.forward(kap, a.N, a.M, a.tau, S);
    ex.backward(c, a.N, a.M, a.tau, dk);
    for (int l = 0; l < a.M; ++l) {
      const int64_t e = e0 + l;
      const float d = dk[l] * a.np.inv_lam;
      if (a.dphi != nullptr) a.dphi[e] = d;
      if (a.phi_out != nullptr) {
        float ph = a.phi[e], m = a.m[e], v = a.v[e];
        adamw_elem(ph, d, m, v, a.opt);
        a.phi_out[e] = ph;
        a.m[e] = m;
        a.v[e] = v;
      }
      if (a.dW != nullptr)
        a.dW[e] = a.hard_in != nullptr
                      ? (((a.hard_in[e >> 5] >> (e & 31)) & 1u) ? a.dWm[e] : uint16_t(0))
                      : __bfloat16_as_ushort(__float2bfloat16_rn(__fmul_rn(bf16_bits_to_float(a.dWm[e]), S[l])));
    }
  }
}

int any_grid(int64_t groups, int per_thread) {
  const int64_t blocks = (groups + int64_t(per_thread) * kThreads - 1) / (int64_t(per_thread) * kThreads);
  const int64_t cap = int64_t(sm_count()) * 32;
  return int(blocks < 1 ? 1 : (blocks < cap ? blocks : cap));
}

}  // namespace

int launch_any_fwd(const FwdCall& c) {
  AnyArgs a{};
  a.phi = c.phi;
  a.W = c.W;
  a.Wm = c.Wm;
  a.soft = c.soft;
  a.hard = c.hard;
  a.st = c.st;
  a.groups = c.E / c.M;
  a.N = c.N;
  a.M = c.M;
  a.tau = c.tau;
  a.inv_tau = 1.0f / c.tau;
  a.np = c.np;
  const bool words = 32 % c.M == 0, exact = !wide_holds(c.N, c.tau);
  if (c.hard != nullptr && (!words || exact)) {
    // assembled with atomicOr
    if (cudaMemsetAsync(c.hard, 0, size_t((c.E + 31) / 32) * 4, c.stream) != cudaSuccess) return -1;
  }
  a.wait = lone_pdl(c.stream);
  int r;
  if (exact) r = launch_maybe_pdl(roi_any_exact_fwd_kernel, any_grid(a.groups, 1), kThreads, 0, c.stream, a.wait, a);
  else if (c.M <= 4) r = launch_maybe_pdl(roi_any_fwd_kernel<4>, any_grid(a.groups, 2), kThreads, 0, c.stream, a.wait, a, words);
  else if (c.M <= 8) r = launch_maybe_pdl(roi_any_fwd_kernel<8>, any_grid(a.groups, 2), kThreads, 0, c.stream, a.wait, a, words);
  else if (c.M <= 16) r = launch_maybe_pdl(roi_any_fwd_kernel<16>, any_grid(a.groups, 1), kThreads, 0, c.stream, a.wait, a, words);
  else r = launch_maybe_pdl(roi_any_fwd_kernel<32>, any_grid(a.groups, 1), kThreads, 0, c.stream, a.wait, a, words);
  return r;
}

int launch_any_bwd(const BwdCall& c) {
  AnyArgs a{};
  a.phi = c.phi;
  a.W = c.W;
  a.dWm = c.dWm;
  a.dphi = c.dphi;
  a.dW = c.dW;
  a.hard_in = c.hard_in;
  a.phi_out = c.phi_out;
  a.m = c.m;
  a.v = c.v;
  a.opt = c.opt;
  a.groups = c.E / c.M;
  a.N = c.N;
  a.M = c.M;
  a.tau = c.tau;
  a.inv_tau = 1.0f / c.tau;
  a.np = c.np;
  const bool exact = !wide_holds(c.N, c.tau);
  a.wait = lone_pdl(c.stream);
  int r;
  if (exact) r = launch_maybe_pdl(roi_any_exact_bwd_kernel, any_grid(a.groups, 1), kThreads, 0, c.stream, a.wait, a);
  else if (c.M <= 4) r = launch_maybe_pdl(roi_any_bwd_kernel<4>, any_grid(a.groups, 2), kThreads, 0, c.stream, a.wait, a);
  else if (c.M <= 8) r = launch_maybe_pdl(roi_any_bwd_kernel<8>, any_grid(a.groups, 2), kThreads, 0, c.stream, a.wait, a);
  else if (c.M <= 16) r = launch_maybe_pdl(roi_any_bwd_kernel<16>, any_grid(a.groups, 1), kThreads, 0, c.stream, a.wait, a);
  else r = launch_maybe_pdl(roi_any_bwd_kernel<32>, any_grid(a.groups, 1), kThreads, 0, c.stream, a.wait, a);
  return r;
}

}  // namespace roi
