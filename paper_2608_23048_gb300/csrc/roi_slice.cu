// Wide groups (M = 16, 32: the 8:16 and 16:32 patterns) on warp slices: the
// SL = M / P consecutive lanes of a slice hold one group, P = 16 members each (8:16: one
// lane, 16:32: two), as packed pairs of neighbouring members (F2).  Each shuffle and tree
// addition then covers more members than with fewer a lane (tau = 0.2, forward + backward
// of 3B-shaped blocks, two at 8:16 and one at 16:32: P = 4 2119 and 2502 us, P = 8 1845
// and 2024, P = 16 1669 and 1684).  Same method as the one-thread-per-group
// kernels (Sec. 4.2.2 Eq. 10-12, Algorithm 1; Eq. 5; backward through the relaxation),
// with the per-group sums and "sum of the other members" formed in the thread and then
// across the slice's lanes by a shuffle that never subtracts.  The step loops
// are rolled: the history of the relaxation that the backward sweeps is indexed in shared
// memory.  Groups whose keys leave the fast path's range are queued by the slice's first
// lane (DeferredGroups) and handled 32 at a time, one per lane, by WideRobustGroup
// (ExactGroup for non-finite keys).
#include <type_traits>

#include "roi_launch.h"
#include "roi_tiles.cuh"

namespace roi {
namespace {

// Launch shapes: threads per CTA (one CTA per SM in either direction), ring stages.
// The backward keeps the last kRegSteps steps of the relaxation in registers and the others in
// shared memory behind the ring (4 P bytes a thread and step).
template <int M>
struct FwdShape {
  static constexpr int kP = 16;  // members of a group per lane
  static constexpr int kThreads = 512;
  static constexpr int kStages = 2;
};
template <int M>
struct BwdShape {
  static constexpr int kP = 16;
  static constexpr int kThreads = M == 16 ? 384 : 256;
  static constexpr int kStages = 1;
  static constexpr int kRegSteps = M == 16 ? 2 : 4;  // last steps of the history kept in registers
};
template <class Shape>
constexpr int kTileOf = Shape::kThreads * Shape::kP;  // elements
template <int N, int M>
constexpr size_t kHistOffset = (tile_smem_bytes<kTileOf<BwdShape<M>>, BwdShape<M>::kStages>(8) + 15) & ~size_t(15);
template <int N, int M>
constexpr size_t kHistBytes = size_t(N - BwdShape<M>::kRegSteps) * BwdShape<M>::kP * sizeof(float) * BwdShape<M>::kThreads;
// Deferred groups: a warp queues at most 32 / SL of them at a time and drains once 32
// are queued.  (3B-shaped set, tau = 0.05, ~4 % of the groups: 8:16 52.8 ms a step with
// the queue against 2424 ms with the routine in place.)
template <int M, class Shape>
constexpr int kDeferCap = 31 + 32 * Shape::kP / M;
template <int M, class Shape>
constexpr size_t kDeferBytes = size_t(kDeferCap<M, Shape>) * 8 * (Shape::kThreads / 32);

template <int M>
constexpr size_t kFwdDeferOffset = (tile_smem_bytes<kTileOf<FwdShape<M>>, FwdShape<M>::kStages>(6) + 15) & ~size_t(15);
template <int N, int M>
constexpr size_t kBwdDeferOffset = (kHistOffset<N, M> + kHistBytes<N, M> + 15) & ~size_t(15);

// The tau != 1 kernels' relaxation: the plain one costs 10 to 15 % less while few groups
// leave its range (8:16, one 11008 x 2048 tensor, forward + backward, plain / WIDE: 254 /
// 291 us at tau = 0.2, 288 / 292 at 0.08, 294 / 292 at 0.06; 16:32: 484 / 562 at 0.2,
// 576 / 560 at 0.1), and at small tau lambda nearly all groups of spread logits do.
constexpr float kSliceWideTau = 0.1f;
constexpr float kSliceWideTauLambda = 0.05f;
__device__ __forceinline__ float shfl_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ F2 swap(F2 v) { return f2(hi(v), lo(v)); }

// Sum of v over the slice's other lanes (never total minus own).
template <int SL>
__device__ __forceinline__ float sum_others(float v) {
  float oth = 0.0f;
#pragma unroll
  for (int o = 1; o < SL; o <<= 1) {
    const float sib = shfl_xor(v, o);
    oth = o == 1 ? sib : __fadd_rn(oth, sib);
    v = __fadd_rn(v, sib);
  }
  return oth;
}
// Sum over the group of a packed per-lane partial.
template <int SL>
__device__ __forceinline__ float group_sum(F2 p) {
  float v = __fadd_rn(lo(p), hi(p));
#pragma unroll
  for (int o = 1; o < SL; o <<= 1) v = __fadd_rn(v, shfl_xor(v, o));
  return v;
}
template <int H>
__device__ __forceinline__ F2 sum_pk(const F2 (&x)[H]) {
  F2 t[H / 2];
#pragma unroll
  for (int i = 0; i < H / 2; ++i) t[i] = x[2 * i] + x[2 * i + 1];
  if constexpr (H == 2) {
    return t[0];
  } else {
    return sum_pk(t);
  }
}
// For every member the sum over the group's other members, and the group's total: the
// pairs' halves are summed in lockstep, and each half's total and the other lanes' enter
// the other half's sums.
template <int SL, int H>
__device__ __forceinline__ float exclusive(const F2 (&x)[H], F2 (&ex)[H]) {
  static_assert(H == 8, "16 members a lane");
  F2 p[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) p[i] = x[2 * i] + x[2 * i + 1];
  const F2 q0 = p[0] + p[1], q1 = p[2] + p[3];
  const F2 t = q0 + q1;
  const float own = __fadd_rn(lo(t), hi(t));
  const float oth = sum_others<SL>(own);
  const F2 beyond = SL == 1 ? swap(t) : swap(t) + f2(oth);
  const F2 r0 = q0 + beyond, r1 = q1 + beyond;
  const F2 e[4] = {p[1] + r1, p[0] + r1, p[3] + r0, p[2] + r0};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    ex[2 * i] = x[2 * i + 1] + e[i];
    ex[2 * i + 1] = x[2 * i] + e[i];
  }
  return SL == 1 ? own : __fadd_rn(own, oth);
}
template <int SL, int H>
__device__ __forceinline__ float group_max(const F2 (&x)[H]) {
  float m = fmaxf(lo(x[0]), hi(x[0]));
#pragma unroll
  for (int i = 1; i < H; ++i) m = fmax3(m, lo(x[i]), hi(x[i]));
#pragma unroll
  for (int o = 1; o < SL; o <<= 1) m = fmaxf(m, shfl_xor(m, o));
  return m;
}
// The group's second largest value (ties count twice).
template <int SL, int H>
__device__ __forceinline__ float group_second(const F2 (&x)[H]) {
  float h[H], s[H];
#pragma unroll
  for (int i = 0; i < H; ++i) h[i] = fmaxf(lo(x[i]), hi(x[i])), s[i] = fminf(lo(x[i]), hi(x[i]));
#pragma unroll
  for (int w = H / 2; w >= 1; w >>= 1) {
#pragma unroll
    for (int i = 0; i < w; ++i) {
      s[i] = fmax3(fminf(h[i], h[i + w]), s[i], s[i + w]);
      h[i] = fmaxf(h[i], h[i + w]);
    }
  }
  float m1 = h[0], m2 = s[0];
#pragma unroll
  for (int o = 1; o < SL; o <<= 1) {
    const float o1 = shfl_xor(m1, o), o2 = shfl_xor(m2, o);
    m2 = fmax3(fminf(m1, o1), m2, o2);
    m1 = fmaxf(m1, o1);
  }
  return m2;
}

struct SliceArgs {
  const float* phi;
  const uint16_t* W;
  const uint16_t* dWm;
  uint16_t* Wm;
  float* soft;
  uint32_t* hard;
  float* dphi;
  uint16_t* dW;
  bool st;                  // straight-through forward: Wm = W where the hard mask is set
  const uint32_t* hard_in;  // straight-through backward: dW = dWm where the forward's bit is set
  float* phi_out;           // fused AdamW: logits updated in place
  float* m;
  float* v;
  AdamW opt;
  int64_t E;
  int64_t full_tiles;
  float tau, inv_tau;
  NoiseParams np;
  unsigned int* status;
  bool wait;  // pdl_begin
};

// Dynamic shared memory of the kernels (tile ring, then the step history, the queues).
extern __shared__ __align__(128) uint8_t roi_slice_smem[];

// Keys (log2 units, t = kappa log2 e) of the 2 H members whose logits are at p and whose
// first has call-flat index e0 (a multiple of 8, as the call's first element is).
template <int H>
__device__ __forceinline__ void lane_keys(const float* p, int64_t e0, const NoiseParams& np, F2 (&kap)[H]) {
  const uint64_t q = (np.e_base + uint64_t(e0)) >> 2;
#pragma unroll
  for (int s = 0; s < H / 2; ++s) {
    const float4 v = reinterpret_cast<const float4*>(p)[s];
    const uint4 x = noise_block_q(np, q + s);
    const F2 half = vconst<F2>(__uint_as_float(0x3f7fffffu));
    kap[2 * s] = key_log2(f2(v.x, v.y), f2(one_plus_from_word(x.x), one_plus_from_word(x.y)) - half, np.l2e_inv_lam);
    kap[2 * s + 1] =
        key_log2(f2(v.z, v.w), f2(one_plus_from_word(x.z), one_plus_from_word(x.w)) - half, np.l2e_inv_lam);
  }
}

// Forward relaxation of the group held by this slice; with KEEP every step's mu is kept
// for backward().  WIDE (tau != 1): as FastGroup's, no finite key leaves the range.
template <int N, int M, int P, bool TAU1, bool KEEP, bool WIDE>
struct SliceRelax {
  static constexpr int SL = M / P;
  static constexpr int kPk = P / 2;
  static constexpr int T = BwdShape<M>::kThreads;
  F2 S[kPk];                 // without KEEP
  // KEEP: mu of the last R steps here, of the others in hist[(k P / 4 + i) T]
  static constexpr int R = BwdShape<M>::kRegSteps;
  F2 keep[KEEP ? R : 1][kPk];
  ulonglong2* hist;

  __device__ __forceinline__ void put(int k, const F2 (&mu)[kPk]) {
#pragma unroll
    for (int i = 0; i < P / 4; ++i) hist[(k * (P / 4) + i) * T] = make_ulonglong2(mu[2 * i].v, mu[2 * i + 1].v);
  }
  __device__ __forceinline__ void get(int k, F2 (&mu)[kPk]) const {
#pragma unroll
    for (int i = 0; i < P / 4; ++i) {
      const ulonglong2 a = hist[(k * (P / 4) + i) * T];
      mu[2 * i].v = a.x, mu[2 * i + 1].v = a.y;
    }
  }
  // KEEP: the soft mask, summed from the history on demand (the backward's optional dW)
  __device__ __forceinline__ void soft(F2 (&s)[kPk]) const {
#pragma unroll
    for (int i = 0; i < kPk; ++i) {
      s[i] = keep[0][i];
#pragma unroll
      for (int j = 1; j < R; ++j) s[i] = s[i] + keep[j][i];
    }
#pragma unroll 1
    for (int k = 0; k < N - R; ++k) {
      F2 mu[kPk];
      get(k, mu);
#pragma unroll
      for (int i = 0; i < kPk; ++i) s[i] = s[i] + mu[i];
    }
  }

  // One step's mu joins the history or the soft mask.
  __device__ __forceinline__ void use(int k, const F2 (&e)[kPk], F2 r) {
    if constexpr (KEEP) {
      F2 mu[kPk];
#pragma unroll
      for (int i = 0; i < kPk; ++i) mu[i] = e[i] * r;
      if (k < N - R) {
        put(k, mu);
      } else {
#pragma unroll
        for (int j = 0; j < R; ++j)
          if (k == N - R + j) {
#pragma unroll
            for (int i = 0; i < kPk; ++i) keep[j][i] = mu[i];
          }
      }
    } else {
#pragma unroll
      for (int i = 0; i < kPk; ++i) S[i] = vfma(e[i], r, S[i]);
    }
  }

  // Returns whether the group left the float range (or has a non-finite key), the same on
  // every lane of the slice.
  __device__ __forceinline__ bool forward(const F2 (&kap)[kPk], float inv_tau, int base_lane) {
    const F2 itau = f2(inv_tau);
    constexpr int kPeel = KEEP ? R : 1;  // steps outside the rolled loop
    bool flag = false;
    F2 x[kPk], e[kPk], ex[kPk];
    if constexpr (!KEEP) {
#pragma unroll
      for (int i = 0; i < kPk; ++i) S[i] = f2(0.0f);
    }
    if constexpr (TAU1) {
      // weights relative to the slice's first key; a member more than 100 log2 units from
      // it (or a non-finite key) sends the group to the exact routine
      const F2 ref = f2(__shfl_sync(0xffffffffu, lo(kap[0]), base_lane));
      float emin = INFINITY;
#pragma unroll
      for (int i = 0; i < kPk; ++i) {
        x[i] = vmap(kap[i] - ref, ex2_approx);
        emin = fminf(emin, fminf(lo(x[i]), hi(x[i])));
      }
      const float tot = group_sum<SL>(sum_pk(x));
      bool out = !(emin >= kTinyExcl) || !(tot <= 1.0f / kTinyExcl);
      flag = (__ballot_sync(0xffffffffu, out) >> base_lane & ((1u << SL) - 1u)) != 0u;
      F2 r = f2(rcp_approx(tot));
      auto step = [&](int k) {
        use(k, x, r);
        if (k + 1 < N) {
          F2 cur[kPk];
#pragma unroll
          for (int i = 0; i < kPk; ++i) cur[i] = x[i] * r;
          exclusive<SL>(cur, ex);
#pragma unroll
          for (int i = 0; i < kPk; ++i) x[i] = cur[i] * ex[i];
          r = f2(rcp_approx(group_sum<SL>(sum_pk(x))));
        }
      };
#pragma unroll 2
      for (int k = 0; k < N - kPeel; ++k) step(k);
#pragma unroll
      for (int k = N - kPeel; k < N; ++k) step(k);
    } else if constexpr (WIDE) {
      float sq = 0.0f;
#pragma unroll
      for (int i = 0; i < kPk; ++i) sq = fmaf(lo(kap[i]), lo(kap[i]), fmaf(hi(kap[i]), hi(kap[i]), sq));
      sq = group_sum<SL>(f2(sq, 0.0f));
      flag = !(sq - sq >= 0.0f);  // a non-finite key, or one beyond 2^63
      const F2 ref = f2(group_second<SL>(kap));
#pragma unroll
      for (int i = 0; i < kPk; ++i) x[i] = (kap[i] - ref) * itau;
      auto step = [&](int k) {
        F2 c[kPk];
#pragma unroll
        for (int i = 0; i < kPk; ++i) {
          c[i] = vmin(x[i], f2(kLeadCap));
          e[i] = vmap(c[i], ex2_approx);
        }
        if (k + 1 < N) {
          const F2 r = f2(rcp_approx(exclusive<SL>(e, ex)));
          use(k, e, r);
#pragma unroll
          for (int i = 0; i < kPk; ++i) x[i] = vfma(vmap(ex[i] * r, lg2_approx) - (x[i] - c[i]), itau, x[i]);
          const F2 m = f2(group_second<SL>(x));
#pragma unroll
          for (int i = 0; i < kPk; ++i) x[i] = x[i] - m;
        } else {
          use(k, e, f2(rcp_approx(group_sum<SL>(sum_pk(e)))));
        }
      };
#pragma unroll 1
      for (int k = 0; k < N - kPeel; ++k) step(k);
#pragma unroll
      for (int k = N - kPeel; k < N; ++k) step(k);
    } else {
      const float kmax = group_max<SL>(kap);
      // Range check, from the totals alone: a leader's complement eps (its share of the
      // total) leaves a next total of at most eps + eps^(1 / tau), so eps times the total,
      // the sum that was formed, is at least 2^-99 while
      // log2 total + max(1, tau) log2 (next total) >= -98, and members that were flushed
      // to zero are below the sum's last bit.
      const float tau1 = fmaxf(1.0f, rcp_approx(inv_tau));
      float lz_prev = 0.0f;
#pragma unroll
      for (int i = 0; i < kPk; ++i) x[i] = (kap[i] - f2(kmax)) * itau;
      auto step = [&](int k) {
#pragma unroll
        for (int i = 0; i < kPk; ++i) e[i] = vmap(x[i], ex2_approx);
        const float tot = k + 1 < N ? exclusive<SL>(e, ex) : group_sum<SL>(sum_pk(e));
        const float lz = lg2_approx(tot);
        flag = flag || !(fmaf(lz, tau1, lz_prev) >= kLeastRange);
        lz_prev = lz;
        const F2 r = f2(rcp_approx(tot));
        use(k, e, r);
        if (k + 1 < N) {
          // offset - log2(total) + log2(1 - mu) / tau: normalised, so that the weights of
          // the next step start from mu
#pragma unroll
          for (int i = 0; i < kPk; ++i) x[i] = vfma(vmap(ex[i] * r, lg2_approx), itau, x[i] - f2(lz));
        }
      };
#pragma unroll 1
      for (int k = 0; k < N - kPeel; ++k) step(k);
#pragma unroll
      for (int k = N - kPeel; k < N; ++k) step(k);
    }
    return flag;
  }

  // After forward() with KEEP: dk = tau dL/dkappa of this lane's members for c = dL/dS (the
  // sweep of FastGroup, with b = dk / tau).
  __device__ __forceinline__ void backward(const F2 (&c)[kPk], float inv_tau, F2 (&b)[kPk]) const {
    static_assert(KEEP, "needs the steps");
    const F2 itau = f2(inv_tau);
    {
      F2 cm[kPk];
#pragma unroll
      for (int i = 0; i < kPk; ++i) cm[i] = c[i] * keep[R - 1][i];
      const F2 cmu = f2(group_sum<SL>(sum_pk(cm)));
#pragma unroll
      for (int i = 0; i < kPk; ++i) b[i] = keep[R - 1][i] * (c[i] - cmu);
    }
    auto sweep = [&](const F2 (&mk)[kPk]) {
      F2 om[kPk], h[kPk], H[kPk];
      exclusive<SL>(mk, om);
      // K = <c, mu> + sum b / tau
      F2 dot = c[0] * mk[0];
#pragma unroll
      for (int i = 1; i < kPk; ++i) dot = vfma(c[i], mk[i], dot);
      const F2 K = f2(group_sum<SL>(vfma(sum_pk(b), itau, dot)));
#pragma unroll
      for (int i = 0; i < kPk; ++i) h[i] = b[i] * vmap(om[i], rcp_approx);
      exclusive<SL>(h, H);
#pragma unroll
      for (int i = 0; i < kPk; ++i) b[i] = vfma(mk[i], vfma(H[i], itau, c[i] - K), b[i]);
    };
#pragma unroll
    for (int j = R - 2; j >= 0; --j) sweep(keep[j]);
#pragma unroll 2
    for (int k = N - R - 1; k >= 0; --k) {
      F2 mk[kPk];
      get(k, mk);
      sweep(mk);
    }
  }
};

// Hard bits of a lane's members: rank of each own key among the group's M keys.
template <int M, int P>
__device__ __forceinline__ uint32_t slice_topn_bits(const float (&kap)[P], int N, int base_lane, int q) {
  constexpr int SL = M / P;
  float kk[P];
  int rank[P];
#pragma unroll
  for (int j = 0; j < P; ++j) kk[j] = fmaxf(kap[j], -INFINITY), rank[j] = 0;
#pragma unroll 1
  for (int qq = 0; qq < SL; ++qq) {
#pragma unroll
    for (int jj = 0; jj < P; ++jj) {
      const float ko = __shfl_sync(0xffffffffu, kk[jj], base_lane + qq);
      const int io = qq * P + jj;
#pragma unroll
      for (int j = 0; j < P; ++j) {
        const int im = q * P + j;
        rank[j] += io < im ? (ko >= kk[j]) : (io > im ? (ko > kk[j]) : 0);
      }
    }
  }
  uint32_t bits = 0;
#pragma unroll
  for (int j = 0; j < P; ++j) bits |= uint32_t(rank[j] < N) << j;
  return bits;
}

// Compare-exchange keeping x[a] >= x[b].
template <int P>
__device__ __forceinline__ void ce_desc(float (&x)[P], int a, int b) {
  const float u = x[a], v = x[b];
  x[a] = fmaxf(u, v);
  x[b] = fminf(u, v);
}
// Sorts x[at .. at + 7] descending (Batcher's odd-even merge network).
template <int P>
__device__ __forceinline__ void sort8_desc(float (&x)[P], int at) {
  auto ce = [&](int a, int b) { ce_desc(x, at + a, at + b); };
  ce(0, 1), ce(2, 3), ce(4, 5), ce(6, 7);
  ce(0, 2), ce(1, 3), ce(4, 6), ce(5, 7);
  ce(1, 2), ce(5, 6);
  ce(0, 4), ce(1, 5), ce(2, 6), ce(3, 7);
  ce(2, 4), ce(3, 5);
  ce(1, 2), ce(3, 4), ce(5, 6);
}
// Sorts a bitonic run x[at .. at + n - 1] descending.
template <int n, int P>
__device__ __forceinline__ void bitonic_desc(float (&x)[P], int at) {
#pragma unroll
  for (int d = n / 2; d >= 1; d >>= 1)
#pragma unroll
    for (int i = 0; i < n; ++i)
      if ((i & d) == 0) ce_desc(x, at + i, at + i + d);
}

// Hard bits of a lane's members for N = M / 2 (the two patterns of these kernels) from the
// group's N-th largest key: each half of the group is sorted (8:16: both in the lane,
// 16:32: one per lane of the slice); the top M / 2 of the group are then the larger
// elements of the pairs (i-th of the first half, i-th from the end of the second), so
// their minimum is the threshold.  A member is kept iff its key reaches it.  Returns false (bits unusable) if
// the slice's keys are not all finite or the threshold is tied, so that more than N
// members pass: the caller ranks such groups by comparison.
template <int N, int M, int P>
__device__ __forceinline__ bool slice_topn_threshold(const float (&kap)[P], uint32_t& bits) {
  static_assert(2 * N == M, "threshold selection needs N = M / 2");
  constexpr int SL = M / P;
  static_assert(P == 16 && SL <= 2, "two runs of eight a lane, at most two lanes a group");
  float x[P];
#pragma unroll
  for (int i = 0; i < P; ++i) x[i] = kap[i];
#pragma unroll
  for (int i = 0; i < P; i += 8) sort8_desc(x, i);
  float m = INFINITY;
  if constexpr (SL == 1) {
#pragma unroll
    for (int i = 0; i < P / 2; ++i) m = fminf(m, fmaxf(x[i], x[P - 1 - i]));
  } else {
    // the lane's two sorted runs into one
#pragma unroll
    for (int i = 0; i < 8; ++i) ce_desc(x, i, 15 - i);
    bitonic_desc<8>(x, 0);
    bitonic_desc<8>(x, 8);
#pragma unroll
    for (int i = 0; i < P; ++i) m = fminf(m, fmaxf(x[i], shfl_xor(x[P - 1 - i], 1)));
  }
  bits = 0;
  float fin = 0.0f;
#pragma unroll
  for (int i = 0; i < P; ++i) {
    bits |= uint32_t(kap[i] >= m) << i;
    fin += kap[i] - kap[i];  // 0 for finite keys, NaN otherwise
  }
  int cnt = __popc(bits) + (fin == 0.0f ? 0 : 64);
#pragma unroll
  for (int o = 1; o < SL; o <<= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  return cnt == N;
}

// Hard bits of a lane's members: the threshold selection, and for a group it cannot
// settle (a tie at the threshold, a non-finite key) comparison ranking, run by the whole
// warp when any of its groups needs it.
template <int N, int M, int H>
__device__ __forceinline__ uint32_t lane_topn(const F2 (&kap)[H], int base_lane, int q) {
  float k[2 * H];
#pragma unroll
  for (int i = 0; i < H; ++i) k[2 * i] = lo(kap[i]), k[2 * i + 1] = hi(kap[i]);
  uint32_t bits;
  const bool ok = slice_topn_threshold<N, M>(k, bits);
  if (__any_sync(0xffffffffu, !ok)) {
    const uint32_t b = slice_topn_bits<M>(k, N, base_lane, q);
    if (!ok) bits = b;
  }
  return bits;
}

// The keys of all M elements of one group, in log2 units, from logits at phi_g
// (call-flat index g0), by one lane.
template <int N, int M>
__device__ __forceinline__ void group_keys_all(const float* phi_g, int64_t g0, const NoiseParams& np, float (&k)[M]) {
#pragma unroll
  for (int s = 0; s < M / 8; ++s) {
    F2 k8[4];
    lane_keys(phi_g + 8 * s, g0 + 8 * s, np, k8);
#pragma unroll
    for (int i = 0; i < 4; ++i) k[8 * s + 2 * i] = lo(k8[i]), k[8 * s + 2 * i + 1] = hi(k8[i]);
  }
}
// The exact relaxation of one group with keys t (log2 units): WideRobustGroup for finite
// keys (which never come here from a WIDE kernel), ExactGroup (natural-log keys) otherwise;
// soft mask S and, with c, dk = dL/dkappa.
template <int N, int M, bool BWD, bool WIDE>
__device__ __forceinline__ void exact_relax(float (&t)[M], const float (&c)[M], const SliceArgs& a, float (&S)[M],
                                            float (&dk)[M]) {
  if (!WIDE && all_finite(t)) {
    WideRobustGroup<N, M> rg;
    rg.forward(t, a.inv_tau, S);
    if constexpr (BWD) rg.backward(c, a.inv_tau, dk);
  } else {
#pragma unroll
    for (int l = 0; l < M; ++l) t[l] *= kLn2;  // natural-log keys
    ExactGroup<N, M> ex;
    ex.forward(t, N, M, a.tau, S);
    if constexpr (BWD) ex.backward(c, N, M, a.tau, dk);
  }
}

__device__ __forceinline__ uint2 pack4(const float (&w)[4], const float (&s)[4]) {
  uint2 o;
  o.x = pack_bf16x2(__fmul_rn(w[0], s[0]), __fmul_rn(w[1], s[1]));
  o.y = pack_bf16x2(__fmul_rn(w[2], s[2]), __fmul_rn(w[3], s[3]));
  return o;
}
__device__ __forceinline__ void unpack_bf16x4(uint2 q, float (&out)[4]) {
  out[0] = bf16_bits_to_float(q.x & 0xffffu);
  out[1] = bf16_bits_to_float(q.x >> 16);
  out[2] = bf16_bits_to_float(q.y & 0xffffu);
  out[3] = bf16_bits_to_float(q.y >> 16);
}

// The exact routine for one group (first element g0, call-flat), from global
// memory: the forward's outputs (Wm unless straight-through, soft).
template <int N, int M, bool WIDE>
__device__ __forceinline__ void exact_group_fwd(int64_t g0, const SliceArgs& a) {
  if (a.soft == nullptr && a.st) return;
  float k[M], S[M], unused[M];
  group_keys_all<N, M>(a.phi + g0, g0, a.np, k);
  exact_relax<N, M, false, WIDE>(k, k, a, S, unused);
#pragma unroll 1
  for (int s = 0; s < M / 4; ++s) {
    float wv[4], sv[4];
    unpack_bf16x4(*reinterpret_cast<const uint2*>(a.W + g0 + 4 * s), wv);
#pragma unroll
    for (int j = 0; j < 4; ++j) sv[j] = S[4 * s + j];
    if (!a.st) *reinterpret_cast<uint2*>(a.Wm + g0 + 4 * s) = pack4(wv, sv);
    if (a.soft != nullptr) *reinterpret_cast<float4*>(a.soft + g0 + 4 * s) = make_float4(sv[0], sv[1], sv[2], sv[3]);
  }
}
// The backward's outputs of one group: dphi, the fused AdamW step, dW unless the
// straight-through variant (which wrote it with the fast path).  The group's logits
// are untouched until here (the fast path skips its AdamW step).
template <int N, int M, bool WIDE>
__device__ __forceinline__ void exact_group_bwd(int64_t g0, const SliceArgs& a) {
  float k[M], cc[M], S[M], dkk[M];
  group_keys_all<N, M>(a.phi + g0, g0, a.np, k);
#pragma unroll 1
  for (int s = 0; s < M / 4; ++s) {
    float wv[4], dv[4];
    unpack_bf16x4(*reinterpret_cast<const uint2*>(a.W + g0 + 4 * s), wv);
    unpack_bf16x4(*reinterpret_cast<const uint2*>(a.dWm + g0 + 4 * s), dv);
#pragma unroll
    for (int j = 0; j < 4; ++j) cc[4 * s + j] = __fmul_rn(dv[j], wv[j]);
  }
  exact_relax<N, M, true, WIDE>(k, cc, a, S, dkk);
#pragma unroll 1
  for (int s = 0; s < M / 4; ++s) {
    const int64_t e = g0 + 4 * s;
    const float g4[4] = {__fmul_rn(dkk[4 * s], a.np.inv_lam), __fmul_rn(dkk[4 * s + 1], a.np.inv_lam),
                         __fmul_rn(dkk[4 * s + 2], a.np.inv_lam), __fmul_rn(dkk[4 * s + 3], a.np.inv_lam)};
    if (a.dphi != nullptr) *reinterpret_cast<float4*>(a.dphi + e) = make_float4(g4[0], g4[1], g4[2], g4[3]);
    if (a.phi_out != nullptr) adamw4(a.phi_out, a.m, a.v, e, *reinterpret_cast<const float4*>(a.phi + e), g4, a.opt);
    if (a.dW != nullptr && a.hard_in == nullptr) {
      float dv[4], sv[4];
      unpack_bf16x4(*reinterpret_cast<const uint2*>(a.dWm + e), dv);
#pragma unroll
      for (int j = 0; j < 4; ++j) sv[j] = S[4 * s + j];
      *reinterpret_cast<uint2*>(a.dW + e) = pack4(dv, sv);
    }
  }
}

// A lane's 2 H members' worth of bf16 at `p` (16-byte aligned).
template <int H>
__device__ __forceinline__ void unpack_lane(const uint16_t* p, F2 (&out)[H]) {
#pragma unroll
  for (int j = 0; j < H / 4; ++j) {
    const uint4 v = reinterpret_cast<const uint4*>(p)[j];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) out[4 * j + i] = f2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xffff0000u));
  }
}
template <int H>
__device__ __forceinline__ void store_lane(uint16_t* p, const F2 (&v)[H]) {
#pragma unroll
  for (int j = 0; j < H; j += 4)
    reinterpret_cast<uint4*>(p)[j / 4] =
        make_uint4(pack_bf16x2(lo(v[j]), hi(v[j])), pack_bf16x2(lo(v[j + 1]), hi(v[j + 1])),
                   pack_bf16x2(lo(v[j + 2]), hi(v[j + 2])), pack_bf16x2(lo(v[j + 3]), hi(v[j + 3])));
}
template <int H>
__device__ __forceinline__ void store_lane(float* p, const F2 (&v)[H]) {
#pragma unroll
  for (int j = 0; j < H; j += 2)
    reinterpret_cast<float4*>(p)[j / 2] = make_float4(lo(v[j]), hi(v[j]), lo(v[j + 1]), hi(v[j + 1]));
}
// Straight-through: the bf16 values of `src` where the bits are set, +0 elsewhere.
template <int P>
__device__ __forceinline__ void keep_lane(uint16_t* dst, const uint16_t* src, uint32_t bits) {
#pragma unroll
  for (int j = 0; j < P / 8; ++j) {
    const uint4 v = reinterpret_cast<const uint4*>(src)[j];
    const uint2 a = keep4(make_uint2(v.x, v.y), bits >> (8 * j)), b = keep4(make_uint2(v.z, v.w), bits >> (8 * j + 4));
    reinterpret_cast<uint4*>(dst)[j] = make_uint4(a.x, a.y, b.x, b.y);
  }
}

// Forward of a lane's members (p, w: their logits and weights in shared or global memory,
// e0: call-flat index of the first).  All 32 lanes call this together; inactive ones
// (ragged tail) take part in the shuffles with zero keys.  Returns whether the group goes
// to the exact routine (on its first lane).
template <int N, int M, int P, bool TAU1, bool WIDE, class Release>
__device__ __forceinline__ bool fwd_lane(const float* p, const uint16_t* w, int64_t e0, bool active, const SliceArgs& a,
                                         const Release& release) {
  constexpr int SL = M / P, kPk = P / 2;
  const int lane = threadIdx.x & 31, q = lane % SL, base_lane = lane - q;
  F2 kap[kPk];
  if (active) {
    lane_keys(p, e0, a.np, kap);
  } else {
#pragma unroll
    for (int i = 0; i < kPk; ++i) kap[i] = f2(0.0f);
  }
  uint32_t bits = 0;
  if (a.hard != nullptr || a.st) bits = lane_topn<N, M>(kap, base_lane, q);
  SliceRelax<N, M, P, TAU1, false, WIDE> rx;
  const bool flag = rx.forward(kap, a.inv_tau, base_lane);
  if (active) {
    if (a.st) {
      keep_lane<P>(a.Wm + e0, w, bits);
    } else if (!flag) {
      F2 m[kPk];
      unpack_lane(w, m);
#pragma unroll
      for (int i = 0; i < kPk; ++i) m[i] = m[i] * rx.S[i];
      store_lane(a.Wm + e0, m);
    }
    if (a.soft != nullptr && !flag) store_lane(a.soft + e0, rx.S);
  }
  release();
  if (a.hard != nullptr) {
    constexpr int kPerWord = 32 / P;
    uint32_t v = active ? bits << ((lane % kPerWord) * P) : 0u;
#pragma unroll
    for (int o = 1; o < kPerWord; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
    if (active && lane % kPerWord == 0) a.hard[e0 >> 5] = v;
  }
  return active && q == 0 && flag;
}

// Backward of a lane's members (as fwd_lane).
template <int N, int M, int P, bool TAU1, bool WIDE, class Release>
__device__ __forceinline__ bool bwd_lane(const float* p, const uint16_t* w, const uint16_t* dw, int64_t e0, bool active,
                                         const SliceArgs& a, const Release& release) {
  constexpr int SL = M / P, kPk = P / 2;
  const int lane = threadIdx.x & 31, q = lane % SL, base_lane = lane - q;
  F2 kap[kPk], c[kPk], b[kPk];
  if (active) {
    lane_keys(p, e0, a.np, kap);
    F2 wv[kPk];
    unpack_lane(w, wv);
    unpack_lane(dw, c);
#pragma unroll
    for (int i = 0; i < kPk; ++i) c[i] = c[i] * wv[i];
  } else {
#pragma unroll
    for (int i = 0; i < kPk; ++i) kap[i] = c[i] = f2(0.0f);
  }
  // the stage is free from here on: its refill lands during the relaxation, so one stage
  // suffices and the shared memory goes to the step history
  release();
  SliceRelax<N, M, P, TAU1, true, WIDE> rx;
  rx.hist = reinterpret_cast<ulonglong2*>(roi_slice_smem + kHistOffset<N, M>) + threadIdx.x;
  const bool flag = rx.forward(kap, a.inv_tau, base_lane);
  if (active && a.dW != nullptr) {
    if (a.hard_in != nullptr) {
      // straight-through: dWm where the forward's hard mask is set
      keep_lane<P>(a.dW + e0, a.dWm + e0, a.hard_in[e0 >> 5] >> (uint32_t(e0) & 31u));
    } else if (!flag) {
      F2 s[kPk], d[kPk];
      rx.soft(s);
      unpack_lane(a.dWm + e0, d);
#pragma unroll
      for (int i = 0; i < kPk; ++i) s[i] = d[i] * s[i];
      store_lane(a.dW + e0, s);
    }
  }
  rx.backward(c, a.inv_tau, b);
  const F2 scale = f2(a.inv_tau * a.np.inv_lam);
#pragma unroll
  for (int i = 0; i < kPk; ++i) b[i] = b[i] * scale;
  if (a.phi_out == nullptr) {
    if (active && !flag) store_lane(a.dphi + e0, b);
  } else {
    // Fused AdamW: the gradients go through this warp's own slots of the step history (read
    // for the last time above), so that consecutive lanes load and store consecutive 16
    // bytes of logits and moments; a lane's own 64 bytes at a time cost the 8:16 backward
    // 25 % (a 67 M element block 996 -> 790 us).  The plain gradients alone are not worth it
    // (16:32, one 3B-shaped block 1664 -> 1750 us).
    ulonglong2* row = rx.hist;
#pragma unroll
    for (int i = 0; i < P / 4; ++i) row[i * BwdShape<M>::kThreads] = make_ulonglong2(b[2 * i].v, b[2 * i + 1].v);
    const uint32_t mine = __ballot_sync(0xffffffffu, active && !flag);
    __syncwarp();
    const int64_t warp_e0 = e0 - int64_t(lane) * P;
#pragma unroll 1
    for (int i = 0; i < P / 4; ++i) {
      const int q4 = i * 32 + lane;  // which four of the warp's members
      const int owner = q4 / (P / 4);
      if ((mine >> owner) & 1u) {
        const float4 g = *reinterpret_cast<const float4*>(row + (q4 % (P / 4)) * BwdShape<M>::kThreads + owner - lane);
        const int64_t e = warp_e0 + 4 * q4;
        if (a.dphi != nullptr) *reinterpret_cast<float4*>(a.dphi + e) = g;
        const float g4[4] = {g.x, g.y, g.z, g.w};
        adamw4(a.phi_out, a.m, a.v, e, *reinterpret_cast<const float4*>(a.phi + e), g4, a.opt);
      }
    }
    __syncwarp();  // the next group's steps go to these slots
  }
  return active && q == 0 && flag;
}

// Runs `lane_fn` for the CTA's full tiles and its chunks of the ragged tail, these straight
// from global memory, queueing the groups it returns true for and handling them by `exact`.
template <int M, class Shape, int NARR, class Exact, class Lane>
__device__ __forceinline__ void slice_walk(const SliceArgs& a, const TileSrc<NARR>& src, size_t defer_at, const Exact& exact,
                                           const Lane& lane_fn) {
  constexpr int kTile = kTileOf<Shape>, P = Shape::kP;
  DeferredGroups<kDeferCap<M, Shape>> dg;
  dg.init(roi_slice_smem + defer_at);
  // a batch's next tensor may start on the SMs this launch frees (no-op otherwise)
  pdl_begin(a.wait);
  const bool ok = run_tiles<Shape::kThreads, kTile, Shape::kStages, NARR>(
      roi_slice_smem, src, a.full_tiles, a.status, [&](const uint8_t* const* stage, int64_t tile, const auto& release) {
        const int64_t e0 = tile * kTile + P * int64_t(threadIdx.x);
        const uint8_t* at[NARR];
#pragma unroll
        for (int i = 0; i < NARR; ++i) at[i] = stage[i] + size_t(P) * src.esize[i] * threadIdx.x;
        dg.push(lane_fn(at, e0, true, release), e0);
        dg.drain(false, exact);
      });
  if (ok) {
    // the ragged tail in warps of lanes, dealt out over the SMs first
    const int64_t t0 = a.full_tiles * kTile;
    const int64_t lanes = (a.E - t0) / P;
    const int lane = threadIdx.x & 31;
    for (int64_t r = 32 * (tail_rank(a.full_tiles) + int64_t(threadIdx.x >> 5) * gridDim.x); r < lanes;
         r += int64_t(gridDim.x) * Shape::kThreads) {
      const bool active = r + lane < lanes;
      const int64_t e0 = t0 + P * (r + lane);
      const uint8_t* at[NARR];
#pragma unroll
      for (int i = 0; i < NARR; ++i) at[i] = src.ptr[i] + (active ? size_t(e0) * src.esize[i] : 0);
      dg.push(lane_fn(at, e0, active, [] {}), e0);
      dg.drain(false, exact);
    }
    dg.drain(true, exact);
  }
  // the launch completes only after the batch's previous one (stream order)
  if (blockIdx.x == 0) pdl_wait();
}

template <int N, int M, bool TAU1, bool WIDE>
__global__ void __launch_bounds__(FwdShape<M>::kThreads, 1) roi_slice_fwd_kernel(SliceArgs a) {
  using C = FwdShape<M>;
  TileSrc<2> src;
  src.ptr[0] = reinterpret_cast<const uint8_t*>(a.phi);
  src.esize[0] = 4;
  src.ptr[1] = reinterpret_cast<const uint8_t*>(a.W);
  src.esize[1] = 2;
  slice_walk<M, C>(a, src, kFwdDeferOffset<M>, [&](int64_t g0) { exact_group_fwd<N, M, WIDE>(g0, a); },
                [&](const uint8_t* const* at, int64_t e0, bool active, const auto& release) {
                  return fwd_lane<N, M, C::kP, TAU1, WIDE>(reinterpret_cast<const float*>(at[0]),
                                                    reinterpret_cast<const uint16_t*>(at[1]), e0, active, a, release);
                });
}

template <int N, int M, bool TAU1, bool WIDE>
__global__ void __launch_bounds__(BwdShape<M>::kThreads, 1) roi_slice_bwd_kernel(SliceArgs a) {
  using C = BwdShape<M>;
  TileSrc<3> src;
  src.ptr[0] = reinterpret_cast<const uint8_t*>(a.phi);
  src.esize[0] = 4;
  src.ptr[1] = reinterpret_cast<const uint8_t*>(a.W);
  src.esize[1] = 2;
  src.ptr[2] = reinterpret_cast<const uint8_t*>(a.dWm);
  src.esize[2] = 2;
  slice_walk<M, C>(a, src, kBwdDeferOffset<N, M>, [&](int64_t g0) { exact_group_bwd<N, M, WIDE>(g0, a); },
                [&](const uint8_t* const* at, int64_t e0, bool active, const auto& release) {
                  return bwd_lane<N, M, C::kP, TAU1, WIDE>(reinterpret_cast<const float*>(at[0]),
                                                    reinterpret_cast<const uint16_t*>(at[1]),
                                                    reinterpret_cast<const uint16_t*>(at[2]), e0, active, a, release);
                });
}

// Multi-tensor launches (a batch's runs of small tensors): the tensors' warps, one after
// another, dealt out over the SMs first; straight from global memory, as the ragged tails.
constexpr int kMultiMax = 192;
struct SliceItem {
  const float* phi;
  const uint16_t* W;
  const uint16_t* dWm;
  uint16_t* Wm;
  float* soft;
  uint32_t* hard;
  float* dphi;
  uint16_t* dW;
  const uint32_t* hard_in;
  float* phi_out;
  float* m;
  float* v;
  int64_t E;
  int64_t tail0;  // first warp of the tensor in the launch
  NoiseParams np;
};
struct SliceMulti {
  int count;
  int64_t total;  // warps
  bool st, wait;
  float tau, inv_tau;
  AdamW opt;
  unsigned int* status;
  SliceItem it[kMultiMax];
};
static_assert(sizeof(SliceMulti) <= 32764, "kernel parameter block");
__device__ __forceinline__ SliceArgs slice_args(const SliceMulti& mm, int i) {
  const SliceItem& x = mm.it[i];
  SliceArgs a;
  a.phi = x.phi, a.W = x.W, a.dWm = x.dWm;
  a.Wm = x.Wm, a.soft = x.soft, a.hard = x.hard;
  a.dphi = x.dphi, a.dW = x.dW, a.hard_in = x.hard_in;
  a.phi_out = x.phi_out, a.m = x.m, a.v = x.v;
  a.st = mm.st;
  a.opt = mm.opt;
  a.E = x.E;
  a.full_tiles = 0;
  a.tau = mm.tau, a.inv_tau = mm.inv_tau;
  a.np = x.np;
  a.status = mm.status;
  a.wait = false;
  return a;
}
template <int M, bool BWD>
using ShapeOf = typename std::conditional<BWD, BwdShape<M>, FwdShape<M>>::type;
template <int N, int M, bool TAU1, bool WIDE, bool BWD>
__global__ void __launch_bounds__(ShapeOf<M, BWD>::kThreads, 1) roi_slice_multi_kernel(const __grid_constant__ SliceMulti mm) {
  using C = ShapeOf<M, BWD>;
  constexpr int P = C::kP;
  constexpr int64_t kLow = (int64_t(1) << 48) - 1;
  DeferredGroups<kDeferCap<M, C>> dg;
  dg.init(roi_slice_smem + (BWD ? kBwdDeferOffset<N, M> : kFwdDeferOffset<M>));
  const auto exact = [&](int64_t e) {
    if constexpr (BWD) {
      exact_group_bwd<N, M, WIDE>(e & kLow, slice_args(mm, int(e >> 48)));
    } else {
      exact_group_fwd<N, M, WIDE>(e & kLow, slice_args(mm, int(e >> 48)));
    }
  };
  pdl_begin(mm.wait);
  const int lane = threadIdx.x & 31;
  for (int64_t w = blockIdx.x + int64_t(threadIdx.x >> 5) * gridDim.x; w < mm.total; w += int64_t(gridDim.x) * (C::kThreads / 32)) {
    const int i = tail_item(mm, w);
    const SliceArgs a = slice_args(mm, i);
    const int64_t l = 32 * (w - mm.it[i].tail0) + lane;
    const bool active = l < a.E / P;
    const int64_t e0 = P * l, at = active ? e0 : 0;
    bool defer;
    if constexpr (BWD) {
      defer = bwd_lane<N, M, P, TAU1, WIDE>(a.phi + at, a.W + at, a.dWm + at, e0, active, a, [] {});
    } else {
      defer = fwd_lane<N, M, P, TAU1, WIDE>(a.phi + at, a.W + at, e0, active, a, [] {});
    }
    dg.push(defer, int64_t(i) << 48 | e0);
    dg.drain(false, exact);
  }
  dg.drain(true, exact);
  // the launch completes only after the batch's previous one (stream order)
  if (blockIdx.x == 0) pdl_wait();
}

// Whether a tau != 1 call takes the WIDE relaxation.
bool slice_wide(int N, float tau, const NoiseParams& np) {
  return wide_holds(N, tau) && (tau < kSliceWideTau || tau < kSliceWideTauLambda * np.inv_lam);
}

struct LaunchCache {
  int per_sm[64] = {0};
};

template <class Shape, class Kern>
int launch_persistent(Kern kern, LaunchCache& cache, size_t smem, SliceArgs a, cudaStream_t stream, bool pdl, bool alone) {
  a.full_tiles = a.E / kTileOf<Shape>;
  a.wait = !pdl && lone_pdl(stream);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  if (cache.per_sm[dev] == 0) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess)
      return -1;
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, Shape::kThreads, smem) != cudaSuccess) return -1;
    cache.per_sm[dev] = per_sm < 1 ? 1 : per_sm;
  }
  const int64_t cap = int64_t(sm_count()) * cache.per_sm[dev];
  // A lone tensor's whole rounds over the SMs go as tiles and the rest, which is all of a small
  // tensor, as its ragged tail, whose warps are spread evenly over the SMs: a lane's sixteen
  // members take N steps one after the other, and the fewer warps share an SM the sooner they
  // are through (8:16 at tau = 0.5 with AdamW, a few tiles more than one round: 24.5 us with
  // those as tiles, 21.5 so; 16:32 straight-through forward of 1.3 M elements 23.2 -> 17.7).
  // A last round that is more than half full stays as tiles, whose loads are staged (8:16
  // forward of 3.7 M elements 19.9 against 20.2 us), but for AdamW's, whose own loads are not
  // (1.8 M elements 30.2 against 26.8).  Where a launch is chained behind, it fills the SMs that
  // the last round leaves (the first tensor of a 3B-shaped set cut: its step 1677 -> 1694 us).
  const int64_t last = a.full_tiles % cap;
  if ((a.full_tiles < cap && !pdl) || (alone && (last <= cap / 2 || a.phi_out != nullptr))) a.full_tiles -= last;
  const int64_t warps = ((a.E - a.full_tiles * kTileOf<Shape>) / Shape::kP + 31) / 32;
  const int64_t want = a.full_tiles + warps;
  const int grid = int(want < 1 ? 1 : (want < cap ? want : cap));
  return launch_maybe_pdl(kern, grid, Shape::kThreads, smem, stream, pdl || a.wait, a);
}

template <int N, int M, bool TAU1, bool WIDE>
int slice_fwd(const SliceArgs& a, cudaStream_t stream, bool pdl, bool alone) {
  static LaunchCache cache;
  constexpr size_t smem = kFwdDeferOffset<M> + kDeferBytes<M, FwdShape<M>>;
  static_assert(smem <= 232448, "shared memory per CTA");
  return launch_persistent<FwdShape<M>>(roi_slice_fwd_kernel<N, M, TAU1, WIDE>, cache, smem, a, stream, pdl, alone);
}
template <int N, int M, bool TAU1, bool WIDE>
int slice_bwd(const SliceArgs& a, cudaStream_t stream, bool pdl, bool alone) {
  static LaunchCache cache;
  constexpr size_t smem = kBwdDeferOffset<N, M> + kDeferBytes<M, BwdShape<M>>;
  static_assert(smem <= 232448, "shared memory per CTA");
  return launch_persistent<BwdShape<M>>(roi_slice_bwd_kernel<N, M, TAU1, WIDE>, cache, smem, a, stream, pdl, alone);
}

template <int N, int M>
int slice_fwd_nm(const SliceArgs& a, cudaStream_t stream, bool pdl, bool alone) {
  if (a.tau == 1.0f) return slice_fwd<N, M, true, false>(a, stream, pdl, alone);
  return slice_wide(N, a.tau, a.np) ? slice_fwd<N, M, false, true>(a, stream, pdl, alone) : slice_fwd<N, M, false, false>(a, stream, pdl, alone);
}
template <int N, int M>
int slice_bwd_nm(const SliceArgs& a, cudaStream_t stream, bool pdl, bool alone) {
  if (a.tau == 1.0f) return slice_bwd<N, M, true, false>(a, stream, pdl, alone);
  return slice_wide(N, a.tau, a.np) ? slice_bwd<N, M, false, true>(a, stream, pdl, alone) : slice_bwd<N, M, false, false>(a, stream, pdl, alone);
}

template <int N, int M, bool TAU1, bool WIDE, bool BWD>
int slice_multi(const SliceMulti& mm, cudaStream_t stream, bool pdl) {
  using C = ShapeOf<M, BWD>;
  static LaunchCache cache;
  constexpr size_t smem = (BWD ? kBwdDeferOffset<N, M> : kFwdDeferOffset<M>) + kDeferBytes<M, C>;
  auto kern = roi_slice_multi_kernel<N, M, TAU1, WIDE, BWD>;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  if (cache.per_sm[dev] == 0) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess) return -1;
    cache.per_sm[dev] = 1;
  }
  const int64_t cap = sm_count();
  const int grid = int(mm.total < 1 ? 1 : (mm.total < cap ? mm.total : cap));
  return launch_maybe_pdl(kern, grid, C::kThreads, smem, stream, pdl || mm.wait, mm);
}
template <int N, int M, bool BWD>
int slice_multi_nm(const SliceMulti& mm, bool wide, cudaStream_t stream, bool pdl) {
  if (mm.tau == 1.0f) return slice_multi<N, M, true, false, BWD>(mm, stream, pdl);
  return wide ? slice_multi<N, M, false, true, BWD>(mm, stream, pdl) : slice_multi<N, M, false, false, BWD>(mm, stream, pdl);
}

void to_item(const FwdCall& c, SliceItem& x) {
  x.Wm = c.Wm;
  x.soft = c.soft;
  x.hard = c.hard;
}
void to_item(const BwdCall& c, SliceItem& x) {
  x.dWm = c.dWm;
  x.dphi = c.dphi;
  x.dW = c.dW;
  x.hard_in = c.hard_in;
  x.phi_out = c.phi_out;
  x.m = c.m;
  x.v = c.v;
}
void to_multi(const FwdCall& c, SliceMulti& mm) { mm.st = c.st; }
void to_multi(const BwdCall& c, SliceMulti& mm) { mm.opt = c.opt; }

// A batch's run of consecutive tensors that shares a launch: at least multi_min_run(false)
// of less than four tiles per SM each, or four of less than one.  One launch per small
// tensor costs its N serial steps each time (16:32, 70 tensors of a few thousand elements:
// 374 -> 31 us forward and backward; 42 of up to 0.8 M: 680 -> 432; the seven of a block of
// 0.4 M at the most: 42 -> 25).  The q, k, v, o tensors between a 3B-shaped block's large
// ones are as fast chained (8:16 forward 317 against 325 us).
template <class Call>
int slice_run(const Call* calls, int count, int64_t tile) {
  const auto run = [&](int64_t tiles_per_sm) {
    int n = 0;
    while (n < count && n < kMultiMax && calls[n].N == calls[0].N && calls[n].M == calls[0].M &&
           calls[n].E < tiles_per_sm * tile * sm_count() &&
           (calls[0].tau == 1.0f || slice_wide(calls[0].N, calls[0].tau, calls[n].np) == slice_wide(calls[0].N, calls[0].tau, calls[0].np)))
      ++n;
    return n;
  };
  const int n = run(4);
  if (n >= multi_min_run(false)) return n;
  const int m = run(1);
  return m >= 4 ? m : 0;
}
template <bool BWD, class Call>
int launch_slice_multi(const Call* calls, int count, bool pdl) {
  static thread_local SliceMulti mm;
  const Call& c0 = calls[0];
  mm.count = count;
  mm.tau = c0.tau;
  mm.inv_tau = 1.0f / c0.tau;
  mm.status = c0.status;
  mm.wait = !pdl && lone_pdl(c0.stream);
  mm.st = false;
  to_multi(c0, mm);
  int64_t warps = 0;
  for (int i = 0; i < count; ++i) {
    SliceItem& x = mm.it[i];
    x = SliceItem{};
    x.phi = calls[i].phi;
    x.W = calls[i].W;
    x.E = calls[i].E;
    x.tail0 = warps;
    x.np = calls[i].np;
    to_item(calls[i], x);
    warps += (calls[i].E / 16 + 31) / 32;
  }
  mm.total = warps;
  const bool wide = slice_wide(c0.N, c0.tau, c0.np);
  if (c0.M == 16) return slice_multi_nm<8, 16, BWD>(mm, wide, c0.stream, pdl);
  return slice_multi_nm<16, 32, BWD>(mm, wide, c0.stream, pdl);
}

}  // namespace

bool slice_supported(int N, int M) { return (N == 8 && M == 16) || (N == 16 && M == 32); }

// The run of small tensors that starts calls[0 .. count) and shares a launch (0: none).
int slice_fwd_run(const FwdCall* calls, int count) {
  return slice_run(calls, count, calls[0].M == 16 ? kTileOf<FwdShape<16>> : kTileOf<FwdShape<32>>);
}
int slice_bwd_run(const BwdCall* calls, int count) {
  return slice_run(calls, count, calls[0].M == 16 ? kTileOf<BwdShape<16>> : kTileOf<BwdShape<32>>);
}
int launch_slice_fwd_multi(const FwdCall* calls, int count, bool pdl) { return launch_slice_multi<false>(calls, count, pdl); }
int launch_slice_bwd_multi(const BwdCall* calls, int count, bool pdl) { return launch_slice_multi<true>(calls, count, pdl); }

int launch_slice_fwd(const FwdCall& c, bool pdl, bool alone) {
  SliceArgs a{};
  a.phi = c.phi;
  a.W = c.W;
  a.Wm = c.Wm;
  a.soft = c.soft;
  a.hard = c.hard;
  a.st = c.st;
  a.E = c.E;
  a.tau = c.tau;
  a.inv_tau = 1.0f / c.tau;
  a.np = c.np;
  a.status = c.status;
  if (c.N == 8 && c.M == 16) return slice_fwd_nm<8, 16>(a, c.stream, pdl, alone);
  if (c.N == 16 && c.M == 32) return slice_fwd_nm<16, 32>(a, c.stream, pdl, alone);
  return -1;
}

int launch_slice_bwd(const BwdCall& c, bool pdl, bool alone) {
  SliceArgs a{};
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
  a.E = c.E;
  a.tau = c.tau;
  a.inv_tau = 1.0f / c.tau;
  a.np = c.np;
  a.status = c.status;
  if (c.N == 8 && c.M == 16) return slice_bwd_nm<8, 16>(a, c.stream, pdl, alone);
  if (c.N == 16 && c.M == 32) return slice_bwd_nm<16, 32>(a, c.stream, pdl, alone);
  return -1;
}

}  // namespace roi
