// Streaming log-softmax kernels over logits rows:
//
//   rl_token_logprobs       logp / entropy / lse of the sampled token per row
//                           (pi(a_t | s_t) of Sec. 2.3; the pi_old recompute of
//                           Sec. 3.2.4)
//   rl_policy_loss_fwd_bwd  the masked clipped objective (Sec. 2.3.1, 2.3.2),
//                           k3-KL, entropy bonus and TIS weight (Sec. 3.2.4), and
//                           d loss / d logits
//
// Design (GB300, sm_103a). Each logits row of the loss kernel is owned by one
// thread-block cluster of C CTAs; CTA k of the cluster takes the k-th slice of the
// row. The slice arrives by bulk asynchronous copies (cp.async.bulk, the 1-D TMA)
// completing on an mbarrier, double-buffered so the copy of the cluster's next row
// overlaps the work on the current one. Pass 1 moves the slice into registers and
// forms an online-softmax partial (max m, sum exp(z - m), sum exp(z - m)(z - m));
// the partials are exchanged through distributed shared memory and merged
// identically in every CTA. Pass 2 writes the gradient from the registers with
// 16-byte stores. Each unmasked row is therefore read from HBM exactly once and its
// gradient written once; masked rows (and rows of trajectories with c_i = 0) are not
// read at all, only zero-filled. A row may start anywhere: it moves in the 16-byte
// blocks of memory that it covers, whatever the leading dimension.
//
// Rows of at most 8 KB (V <= 4,096 bf16 or 2,048 fp32) take a lighter form of the
// loss kernel, a warp per row with the row held in registers (small_rows_kernel).
// The forward-only kernel streams rows through CTAs without clusters
// (stream_logprobs_kernel), short ones through warps (small_logprobs_kernel).
//
// The kernels are persistent: the grid holds as many clusters as fit on the
// GPU at once, and cluster j processes rows j, j + n_clusters, ... . Each
// cluster adds its rows' loss contributions in row order and leaves one partial
// in the workspace; the last cluster to finish (a counter in the workspace
// header) sums the partials in a fixed order into the caller's total, so the
// loss is bit-reproducible without a second launch.
#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "rl_device.cuh"
#include "rl_host.h"

namespace rl {

struct RowArgs {
  const void* logits;
  void* grad;
  int64_t rows, V, ld;
  const int32_t* token_ids;
  const uint8_t* mask;
  const int32_t* token_traj;
  int32_t n_traj;
  const float* adv;
  const float* coef;
  const float* old_logp;
  const float* ref_logp;
  const float* rollout_logp;
  float clip_lo, clip_hi;  // 1 - eps_low, 1 + eps_high
  float beta;              // 0 when the KL term is off
  float alpha;             // entropy bonus
  float tis_cap;           // <= 0 when TIS is off
  int32_t adv_per_row;     // adv holds one A_t per row (else one per trajectory)
  double* row_loss;
  double* loss_accum;      // the caller's total (loss kernel: the last cluster adds into it)
  uint32_t* done;          // finished-cluster count in the workspace header
  float* token_stats;
  float* logp_out;
  float* entropy_out;
  float* lse_out;
  int32_t* status;
  int64_t slice;      // elements per CTA slice, a multiple of the 16-byte vector
  int64_t buf_elems;  // element stride between the two shared-memory buffers
};

// Where a row lies among the 16-byte blocks of the logits (and of the gradient, which has the same
// leading dimension and starts on a 16-byte boundary too). A row may start and end inside a block:
// `head` elements before its first whole block, `vecs` whole blocks, `tail` elements after them.
// Rows of any leading dimension so move in 16-byte blocks, and only the at most
// 2 (16 / sizeof(T) - 1) elements of the two partial blocks go one by one.
template <typename T>
struct RowSpan {
  int head, vecs, tail;
};
template <typename T>
__device__ __forceinline__ RowSpan<T> row_span(int64_t r, int64_t ld, int64_t V) {
  constexpr int EPV = 16 / static_cast<int>(sizeof(T));
  const int off = static_cast<int>(static_cast<uint32_t>(r) * static_cast<uint32_t>(ld)) & (EPV - 1);
  RowSpan<T> s;
  s.head = min((EPV - off) & (EPV - 1), static_cast<int>(V));
  s.vecs = (static_cast<int>(V) - s.head) / EPV;
  s.tail = static_cast<int>(V) - s.head - s.vecs * EPV;
  return s;
}

#ifndef RL_STORE_CS
#define RL_STORE_CS 0
#endif

// 16-byte global store; with RL_STORE_CS the line is marked evict-first (streaming)
__device__ __forceinline__ void st_global_16(void* p, uint4 w) {
#if RL_STORE_CS
  asm volatile("st.global.cs.v4.b32 [%0], {%1, %2, %3, %4};" :: "l"(p), "r"(w.x), "r"(w.y), "r"(w.z), "r"(w.w)
               : "memory");
#else
  *reinterpret_cast<uint4*>(p) = w;
#endif
}

template <typename T>
struct Vec;
template <>
struct Vec<uint16_t> {  // bf16
  static constexpr int N = 8;
  static constexpr int NP = 4;  // float2 pairs per 16-byte vector
  // pad of register-held vectors past the slice: two bf16 values of about -1.5e38, at or below
  // -1e38 (so they count as -inf for the maximum) yet far enough from -FLT_MAX that
  // z log2(e) - m log2(e) stays finite: its exponential is 0 and, with the entropy on, e x is
  // 0, not 0 x -inf = NaN (which would send every thread holding a pad down the slow path)
  static constexpr uint32_t kPadWord = 0xFEE1FEE1u;
  static __device__ __forceinline__ void pairs(const uint4 w, float2 (&q)[4]) {
    q[0] = make_float2(bf16_lo(w.x), bf16_hi(w.x)); q[1] = make_float2(bf16_lo(w.y), bf16_hi(w.y));
    q[2] = make_float2(bf16_lo(w.z), bf16_hi(w.z)); q[3] = make_float2(bf16_lo(w.w), bf16_hi(w.w));
  }
  static __device__ __forceinline__ uint4 pack_pairs(const float2 (&o)[4]) {
    return make_uint4(pack_bf16x2(o[0].x, o[0].y), pack_bf16x2(o[1].x, o[1].y), pack_bf16x2(o[2].x, o[2].y),
                      pack_bf16x2(o[3].x, o[3].y));
  }
  static __device__ __forceinline__ void store_scalar(uint16_t* dst, float g) { *dst = f32_to_bf16(g); }
  static __device__ __forceinline__ float to_f(uint16_t x) { return bf16_to_f32(x); }
};
template <>
struct Vec<float> {
  static constexpr int N = 4;
  static constexpr int NP = 2;
  static constexpr uint32_t kPadWord = 0xFEE1B1E6u;  // -1.5e38: see Vec<uint16_t>::kPadWord
  static __device__ __forceinline__ void pairs(const uint4 w, float2 (&q)[2]) {
    q[0] = make_float2(__uint_as_float(w.x), __uint_as_float(w.y));
    q[1] = make_float2(__uint_as_float(w.z), __uint_as_float(w.w));
  }
  static __device__ __forceinline__ uint4 pack_pairs(const float2 (&o)[2]) {
    return make_uint4(__float_as_uint(o[0].x), __float_as_uint(o[0].y), __float_as_uint(o[1].x),
                      __float_as_uint(o[1].y));
  }
  static __device__ __forceinline__ void store_scalar(float* dst, float g) { *dst = g; }
  static __device__ __forceinline__ float to_f(float x) { return x; }
};

#define RL_NEG_INF (-__int_as_float(0x7f800000))

// Pass 1: -inf (and anything below -1e30) becomes -1e30, so that e = 0 and e (z - m) = 0
// instead of NaN; a NaN stays NaN (a comparison, not fmaxf, which would drop it) and poisons
// its row. Pass 2 clamps with fmaxf: there p = 2^(NaN) is NaN already.
__device__ __forceinline__ float clamp_ninf(float z) { return z < -1e30f ? -1e30f : z; }
constexpr uint32_t kBulkChunk = 32768;

// Elements of src's address past the 16-byte boundary below it.
template <typename T>
__device__ __forceinline__ int block_offset(const T* src) {
  return static_cast<int>((reinterpret_cast<uintptr_t>(src) & 15u) / sizeof(T));
}

template <typename T>
__device__ __forceinline__ bool block_inside(const T* src, const T* end) {
  return src - block_offset(src) + 16 / sizeof(T) <= end;
}

// fold one value into a per-thread online-softmax partial whose max is already >= z
template <bool ENT>
__device__ __forceinline__ void accumulate(SoftmaxPartial& ps, float z, float neg_m_l2e) {
  if (ENT) {
    const float t = clamp_ninf(z) - ps.m;  // -inf logits contribute 0, not NaN
    const float e = ex2(t * kLog2e);
    ps.s += e;
    ps.u = fmaf(e, t, ps.u);
  } else {
    ps.s += ex2(fmaf(z, kLog2e, neg_m_l2e));
  }
}

template <bool ENT>
__device__ __forceinline__ void raise_max(SoftmaxPartial& ps, float vm) {
  if (vm > ps.m) {
    const float d = ps.m - vm;
    const float sc = ex2(d * kLog2e);
    if (ENT) ps.u = (ps.s == 0.f) ? 0.f : sc * fmaf(d, ps.s, ps.u);
    ps.s *= sc;
    ps.m = vm;
  }
}

// Shared-memory stages per CTA (tuning knob). The consumer warps per CTA, the 16-byte vectors
// of the slice each consumer thread holds in registers, the CTAs per SM and the slice size that
// picks the cluster width are chosen per row length on the host (kPicksBf16, kPicksF32).
#ifndef RL_STAGES
#define RL_STAGES 2
#endif

constexpr int kMaxCluster = 16;
// zero-filled shared region, source of the masked rows' bulk stores (8 KB at 2 CTAs per SM:
// 12.947 against 13.029 ms per benchmark step with 2 KB)
constexpr int kZeroBytesMax = 8192;

// Per-row inputs, staged in shared memory by the producer warp. Places in the row are worked out
// there too, once per row and CTA: the consumers' registers are full.
struct RowMeta {
  int64_t r;         // row index, -1 = end of the stream
  int64_t base;      // element offset of this CTA's vector 0 in the gradient
  int32_t nv;        // vectors of this CTA
  int32_t shift;     // fp32: elements of the stage before vector 0
  // elements outside the vectors, one per lane: e_n & 15 of them by the first consumer warp, from
  // e_at in the stage to e_rel after `base`; e_n >> 4 by the second, from the stage's last block to
  // the end of the vectors
  int32_t e_n, e_at, e_rel;
  int32_t a_at;      // the sampled token's place in the stage, -1: another CTA holds it
  int32_t a_rel;     // the same relative to `base`
  int32_t a_writer;  // the thread that stores its gradient, -1: another CTA's
  float A, c, old, ref, roll;
};

// Warp-specialised, cluster-per-row kernel.
//
//   warp NW (producer): walks this cluster's rows cid, cid + ncl, ...; decides which
//     are trained on; zero-fills the others with bulk stores from a zeroed shared
//     region; for a trained row stages its metadata and bulk-copies this CTA's slice
//     into the next free stage (full / empty mbarrier pair per stage).
//   warps 0..NW-1 (consumers): per row, pass 1 over the slice gives one online-softmax
//     partial per warp; every warp pushes its partial to all C CTAs of the cluster
//     with st.async (remote store + complete_tx on the receiver's mailbox mbarrier);
//     each warp then merges all C * NW partials in a fixed order (bit-identical in
//     every warp of every CTA), computes the row's scalars and runs pass 2 (gradient
//     from the registers). The stage is released as soon as the slice is in registers.
// Nothing per row synchronises a whole CTA or the whole cluster.

// Fold NV register-held 16-byte vectors into a partial, branch-free in the common
// case. Vectors past the end of the data hold about -1.5e38 (Vec<T>::kPadWord), whose
// exponential is exactly 0. The reference is the partial's own maximum or, for a
// fresh partial, the first vector's maximum; when the exponentials sum above 1e30
// (a value far above the reference) everything is redone against the exact
// maximum. Values at or below -1e38 count as -inf.
template <typename T, bool ENT, int NV, bool NAN_REF = true, typename Reload>
__device__ __forceinline__ void fold_block(SoftmaxPartial& ps, const uint4 (&x)[NV], Reload reload) {
  constexpr int NP = Vec<T>::NP;
  // NAN_REF: NaN if any value is, so that a thread that has nothing but NaNs (and -inf) takes one as its
  // reference, which poisons the sums; else the largest of the others
  auto larger = [](float a, float b) { return NAN_REF ? max_nan(a, b) : fmaxf(a, b); };
  auto vmax = [&](const uint4 w) {
    float2 q[NP];
    Vec<T>::pairs(w, q);
    float m = larger(q[0].x, q[0].y);
#pragma unroll
    for (int i = 1; i < NP; ++i) m = larger(m, larger(q[i].x, q[i].y));
    return m;
  };
  // exact maximum, recomputed from shared memory (the rare paths only)
  auto all_max = [&]() {
    float m = vmax(reload(0));
    for (int k = 1; k < NV; ++k) m = larger(m, vmax(reload(k)));
    return m;
  };
  if (!(ps.m > -1e38f)) {
    float m0 = vmax(x[0]);
    if (!(m0 > -1e38f)) m0 = all_max();
    if (NAN_REF ? m0 <= -1e38f : !(m0 > -1e38f)) return;
    ps.m = m0;
  }
  // x = (z - m) log2(e) by one fused multiply-add against nm = fl(-m log2(e)); with the
  // entropy, u accumulates e x (log2 units, scaled by ln 2 at the end). A logit at -inf gives
  // e = 0 and e x = NaN: such a block is redone on the clamped path (CLAMP), where z counts as
  // -1e30 (a NaN stays NaN). The rounding of nm shifts every x of the block by the same
  // err = -m log2(e) - nm (exact by one fma); the block's sums are corrected for it once at
  // the end.
  auto exps = [&](auto clamp, const uint4 w, float2& s0, float2& s1, float2& u0) {
    constexpr bool CLAMP = decltype(clamp)::value;
    const float nm = -ps.m * kLog2e;
    const float2 l2 = make_float2(kLog2e, kLog2e), nm2 = make_float2(nm, nm);
    float2 q[NP];
    Vec<T>::pairs(w, q);
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      const float2 qi = CLAMP ? make_float2(clamp_ninf(q[i].x), clamp_ninf(q[i].y)) : q[i];
      const float2 xx = __ffma2_rn(qi, l2, nm2);
      const float2 e = make_float2(ex2(xx.x), ex2(xx.y));
      if (i & 1) s1 = __fadd2_rn(s1, e); else s0 = __fadd2_rn(s0, e);
      if (ENT) u0 = __ffma2_rn(e, xx, u0);
    }
  };
  using Fast = std::integral_constant<bool, false>;
  using Clamped = std::integral_constant<bool, true>;
  const float2 z2 = make_float2(0.f, 0.f);
  float2 s0 = z2, s1 = z2, u0 = z2;
#pragma unroll
  for (int k = 0; k < NV; ++k) exps(Fast{}, x[k], s0, s1, u0);
  float2 sacc = __fadd2_rn(s0, s1);
  float se = sacc.x + sacc.y;
  float ue = ENT ? u0.x + u0.y : 0.f;
  if (!(se <= 1e30f) || (ENT && ue != ue)) {
    // rare: a value far above the reference (move it up to the exact maximum) or a logit at
    // -inf with the entropy on; redo from shared memory on the clamped path
    if (!(se <= 1e30f)) raise_max<ENT>(ps, all_max());
    s0 = z2; s1 = z2; u0 = z2;
    for (int k = 0; k < NV; ++k) exps(Clamped{}, reload(k), s0, s1, u0);
    sacc = __fadd2_rn(s0, s1);
    se = sacc.x + sacc.y;
    ue = ENT ? u0.x + u0.y : 0.f;
  }
  // e_true = e 2^err and x_true = x + err, with |err| <= 2^-24 |m log2(e)|: first order in err
  const float nm = -ps.m * kLog2e;
  const float err = fmaf(-ps.m, kLog2e, -nm);
  const float f = fmaf(err, kLn2, 1.f);
  if (ENT) ps.u = fmaf(fmaf(err, se, ue) * f, kLn2, ps.u);
  ps.s = fmaf(se, f, ps.s);
}

// Log-sum-exp of a row's merged partial as hi + lo. SPLIT: lo is what the rounding of m + ln S and
// of the logarithm leave out (the latter from S e^-lnS = 1 + it), so that the ratio exp(logp - old) is
// off by the error of S alone; without it lo = 0 and the order of operations is the plain one.
struct RowLse {
  float lnS, hi, lo;
};
template <bool SPLIT>
__device__ __forceinline__ RowLse row_lse(const SoftmaxPartial& q) {
  RowLse l{logf(q.s), 0.f, 0.f};
  l.hi = q.m + l.lnS;
  if constexpr (SPLIT) {
    const float b = l.hi - q.m;
    l.lo = (q.m - (l.hi - b)) + (l.lnS - b) + fmaf(q.s, expf(-l.lnS), -1.f);
  }
  return l;
}

// logp - old: large operands are differenced first. SPLIT: with what the rounding of z_a - old leaves
// out, which is up to 5e-7 where the log-prob is about -10. With row_lse's lo the loss of 512 rows of
// 4,096 bf16 entries, a sum that nearly cancels, is off by 1.2e-6 on average over 60 seeds (4.6e-6
// without either), and the gradient of fp32 rows of 151,936 entries by 1.9e-7 (5.0e-7).
template <bool SPLIT>
__device__ __forceinline__ float log_ratio(float za, float old, const RowLse& l) {
  const float d = za - old;
  if constexpr (SPLIT) {
    const float b = d - za;
    const float rest = (za - (d - b)) - (old + b);
    const float x = (d - l.hi) + (rest - l.lo);
    return fabsf(rest) <= 1.f ? x : (d - l.hi) - l.lo;  // infinities leave no rest
  } else {
    return (d - l.hi) - l.lo;
  }
}

// The warp's 32 partials of a row of the loss kernels. bf16: the short chain. fp32: by pairs, whose
// order the results of the fp32 path keep to the bit: a near-one-hot row's gradient is c g (1 - p) at
// the sampled token, so the last bit of a log-sum-exp of 40 (4e-6) shows in it, and the fp32 edge
// batch, bound by HBM, gains nothing from the shorter chain (1,067 us without it, 1,109 us with it).
template <typename T, bool ENT>
__device__ __forceinline__ SoftmaxPartial merge_lanes(SoftmaxPartial p) {
  if constexpr (sizeof(T) == 2) return warp_merge<ENT>(p);
  else return warp_merge_pairs(p);
}

// MINB: CTAs per SM the register budget is sized for (2, or 3 with a smaller zero region).
//
// How a row is cut. bf16: into the 16-byte blocks of memory it covers, CTA k taking blocks
// [k SV, (k + 1) SV) after the row's head, so that a vector is a block wherever the row starts; the
// head's and the tail's elements go one per lane. fp32: into elements, CTA k taking [k slice, (k + 1)
// slice), four to a vector, whatever the row's alignment, so that the order of the sums does not
// depend on it; with SHIFT (a leading dimension that is no multiple of four) a row starts
// `shift` elements into its first block, a vector is read from two blocks, and its gradient is put
// together to whole blocks by shuffles between neighbouring lanes.
template <typename T, int NW, bool ENT, int HOLDV, int MINB, bool SHIFT>
__global__ void __launch_bounds__((NW + 1) * 32, MINB) rows_kernel(const RowArgs p) {
  constexpr bool kBlocks = sizeof(T) == 2;
  static_assert(!(kBlocks && SHIFT), "bf16 rows are cut into blocks");
  constexpr bool kSplit = kBlocks || NW >= 16;  // not where fp32 keeps its bits (merge_lanes)
  constexpr int kZeroBytes = MINB >= 3 ? 2048 : kZeroBytesMax;
  constexpr int EPV = Vec<T>::N;
  constexpr int NB = RL_STAGES;
  constexpr int NC = NW * 32;  // consumer threads
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[NB], empty_bar[NB], xbar[2];
  // twice as deep as the stages: a row's entry is rewritten 2 NB rows on, when every consumer has
  // released the stage of the row NB on and so is done with this one; it can be read (and not held
  // in registers) to the row's end
  __shared__ RowMeta meta[2 * NB];
  __shared__ __align__(16) float4 mbox[2][kMaxCluster * NW];
  __shared__ __align__(128) uint4 zeros[kZeroBytes / 16];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_ctarank(), C = cluster_nctarank();
  const int64_t cid = blockIdx.x / C, ncl = gridDim.x / C;
  const int64_t rows = p.rows, V = p.V, ld = p.ld;
  const int SV = static_cast<int>(p.slice / EPV);
  const int s0 = static_cast<int>(rank) * SV;  // my first block (bf16) or vector (fp32)
  const T* logits = static_cast<const T*>(p.logits);
  const T* const logits_end = logits + ((rows - 1) * ld + V);
  T* grad = static_cast<T*>(p.grad);
  T* const buf_base = reinterpret_cast<T*>(smem_raw);
  // a stage: bf16, the CTA's blocks, the head's block, the tail's; fp32, the blocks that its slice
  // covers (one more than SV where the row starts inside a block)
  const int edge0 = SV * EPV;
  // fp32: a CTA has the same elements of every row, known before its words arrive
  const int n32 = kBlocks ? 0 : max(0, min(static_cast<int>(p.slice), static_cast<int>(V) - s0 * EPV));

  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      mbar_init(&full_bar[k], 1);
      mbar_init(&empty_bar[k], NW);
    }
    mbar_init(&xbar[0], C == 1 ? NW : 1);
    mbar_init(&xbar[1], C == 1 ? NW : 1);
    fence_mbar_init();
  }
  for (int k = tid; k < kZeroBytes / 16; k += blockDim.x) zeros[k] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  __syncthreads();
  if (C > 1) cluster_sync_all();  // every peer's mailbox barrier exists before the first st.async

  if (warp == NW) {
    // =============================================================== producer warp
    // Row metadata is fetched 32 rows at a time, one row per lane, and handed row by row to the
    // staging loop with shuffles. The loads of the next batch are issued while the current one
    // is staged (its owners' coefficients once the owners have arrived), so their latency is
    // hidden behind the copies.
    uint32_t it = 0;
    bool failed = false, stored = false;
    struct Batch {
      int32_t a, i;
      uint32_t m;
      float c, A, old, ref, roll;
    };
    auto load_primary = [&](int64_t b0, Batch& q) {
      const int64_t my = b0 + static_cast<int64_t>(lane) * ncl;
      q = Batch{0, -1, 0u, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (my < rows) {
        q.a = p.token_ids[my];
        q.m = p.mask[my];
        q.i = p.token_traj[my];
        q.old = p.old_logp[my];
        if (p.ref_logp) q.ref = p.ref_logp[my];
        if (p.rollout_logp) q.roll = p.rollout_logp[my];
        if (p.adv_per_row) q.A = p.adv[my];
      }
    };
    auto load_dependent = [&](Batch& q) {
      if (q.m != 0 && q.i >= 0 && q.i < p.n_traj) {
        q.c = p.coef[q.i];
        if (!p.adv_per_row) q.A = p.adv[q.i];
      }
    };
    Batch cur, nxt = Batch{0, -1, 0u, 0.f, 0.f, 0.f, 0.f, 0.f};
    load_primary(cid, cur);
    load_dependent(cur);
    for (int64_t base = cid; base < rows && !failed; base += 32 * ncl) {
      const int64_t next_base = base + 32 * ncl;
      const bool has_next = next_base < rows;
      if (has_next) load_primary(next_base, nxt);
      const int32_t la = cur.a, li = cur.i;
      const uint32_t lm = cur.m;
      const float lc = cur.c, lA = cur.A, lold = cur.old, lref = cur.ref, lroll = cur.roll;
      const int nb = static_cast<int>(min(static_cast<int64_t>(32), (rows - base + ncl - 1) / ncl));
      for (int jr = 0; jr < nb && !failed; ++jr) {
        if (jr == 1 && has_next) load_dependent(nxt);  // the next batch's owners have arrived by now
        const int64_t r = base + static_cast<int64_t>(jr) * ncl;
        RowMeta m;
        m.r = r;
        const int32_t tok = __shfl_sync(0xffffffffu, la, jr);
        bool active = __shfl_sync(0xffffffffu, lm, jr) != 0;
        if (active) {
          const int32_t i = __shfl_sync(0xffffffffu, li, jr);
          if (i < 0 || i >= p.n_traj) {
            if (rank == 0 && lane == 0) flag_status(p.status, RL_DEV_BAD_TRAJ);
            active = false;
          } else {
            m.c = __shfl_sync(0xffffffffu, lc, jr);
            m.A = __shfl_sync(0xffffffffu, lA, jr);
            active = m.c != 0.f;
            if (active && (tok < 0 || tok >= V)) {
              if (rank == 0 && lane == 0) flag_status(p.status, RL_DEV_BAD_TOKEN);
              active = false;
            }
          }
        }
        const T* row = logits + r * ld;
        // this CTA's part of the gradient row as whole 16-byte blocks, `pre` elements before them and
        // `post` after them
        RowSpan<T> span;
        int64_t first;  // element offset of the first of those blocks
        int pre, blocks, post;
        if constexpr (kBlocks) {
          span = row_span<T>(r, ld, V);
          blocks = max(0, min(SV, span.vecs - s0));
          pre = rank == 0 ? span.head : 0;
          post = rank == C - 1 ? span.tail : 0;
          first = r * ld + span.head + static_cast<int64_t>(s0) * EPV;
        } else {
          m.shift = SHIFT ? block_offset(row) : 0;
          pre = SHIFT ? min(n32, (EPV - m.shift) & (EPV - 1)) : 0;
          blocks = (n32 - pre) / EPV;
          post = n32 - pre - blocks * EPV;
          first = r * ld + s0 * EPV + pre;
        }
        if (!active) {
          // zero it
          const uint32_t bytes = static_cast<uint32_t>(blocks) * 16u;
          if (lane == 0 && bytes > 0) {
            char* g = reinterpret_cast<char*>(grad + first);
            for (uint32_t off = 0; off < bytes; off += kZeroBytes)
              bulk_s2g(g + off, zeros, min(static_cast<uint32_t>(kZeroBytes), bytes - off));
            bulk_commit();
            stored = true;
          }
          if (lane < pre) grad[first - pre + lane] = T(0);
          if (lane < post) grad[first + static_cast<int64_t>(blocks) * EPV + lane] = T(0);
          if (rank == 0 && lane == 0 && p.token_stats)
            for (int k = 0; k < 5; ++k) p.token_stats[r * 5 + k] = 0.f;
          continue;
        }
        m.old = __shfl_sync(0xffffffffu, lold, jr);
        m.ref = __shfl_sync(0xffffffffu, lref, jr);
        m.roll = __shfl_sync(0xffffffffu, lroll, jr);
        // what to copy: `copy_bytes` from `src` to the stage's start, and up to two lone elements'
        // blocks: a bulk copy of 16 bytes each, or, where the block reaches past the end of the
        // logits (at the last row), its elements one by one. All of this is worked out before the
        // wait for the stage.
        const int b = it % NB;
        T* buf = buf_base + b * p.buf_elems;
        const T* src;
        uint32_t copy_bytes, lone_bytes = 0;
        const T *lone[2] = {row, row};         // blocks copied on their own (bf16: head, tail)
        bool lone_bulk[2] = {false, false};
        const T* by_one = row;                 // elements copied one by one, and where to
        int by_one_n = 0, by_one_at = 0;
        m.a_at = m.a_writer = -1;
        if constexpr (kBlocks) {
          const int hoff = block_offset(row);
          const T* tail = row + (V - span.tail);
          src = logits + first;
          copy_bytes = static_cast<uint32_t>(blocks) * 16u;
          lone[0] = row - hoff;
          lone[1] = tail;
          lone_bulk[0] = pre > 0 && block_inside(row, logits_end);
          lone_bulk[1] = post > 0 && block_inside(tail, logits_end);
          if (post > 0 && !lone_bulk[1]) {
            by_one = tail;
            by_one_n = post;
            by_one_at = edge0 + EPV;
          } else if (pre > 0 && !lone_bulk[0]) {  // a row shorter than a block: no tail
            by_one = row;
            by_one_n = pre;
            by_one_at = edge0 + hoff;
          }
          m.base = first;
          m.nv = blocks;
          m.shift = 0;
          m.e_n = pre | post << 4;
          m.e_at = edge0 + hoff;
          m.e_rel = -pre;
          m.a_rel = tok - span.head - s0 * EPV;
          const int tail0 = static_cast<int>(V) - span.tail;  // the tail's first element
          if (tok < span.head) {
            if (rank == 0) {
              m.a_at = edge0 + hoff + tok;
              m.a_writer = tok;
            }
          } else if (tok >= tail0) {
            if (rank == C - 1) {
              m.a_at = edge0 + EPV + (tok - tail0);
              m.a_writer = 32 + (tok - tail0);
            }
          } else if (m.a_rel >= 0 && m.a_rel < blocks * EPV) {
            m.a_at = m.a_rel;
            m.a_writer = m.a_rel / EPV % NC;
          }
        } else {
          const int d = m.shift;
          src = row + s0 * EPV - d;
          int nblk = (d + n32 + EPV - 1) / EPV;
          if (n32 <= 0) nblk = 0;
          if (src + static_cast<int64_t>(nblk) * EPV > logits_end && nblk > 0) {
            --nblk;
            by_one = src + nblk * EPV;
            by_one_n = d + n32 - nblk * EPV;
            by_one_at = nblk * EPV;
          }
          copy_bytes = static_cast<uint32_t>(nblk) * 16u;
          m.base = r * ld + s0 * EPV;
          m.nv = n32 / EPV;
          m.e_n = n32 % EPV;
          m.e_at = d + m.nv * EPV;
          m.e_rel = m.nv * EPV;
          m.a_rel = tok - s0 * EPV;
          if (m.a_rel >= 0 && m.a_rel < n32) {
            m.a_at = d + m.a_rel;
            // the thread whose store covers it: its vector's, or, for the elements before a block
            // boundary inside it, the lane before that one
            const int t = m.a_rel / EPV % NC;
            m.a_writer = m.a_rel >= m.nv * EPV ? m.a_rel - m.nv * EPV
                         : SHIFT && d != 0 && m.a_rel % EPV < EPV - d && t % 32 != 0 ? t - 1 : t;
          }
        }
        if (lone_bulk[0]) lone_bytes += 16u;
        if (lone_bulk[1]) lone_bytes += 16u;
        const uint32_t use = it / NB;
        if (use > 0 && !mbar_wait_bounded(&empty_bar[b], (use - 1) & 1)) {
          failed = true;
          if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
          break;
        }
        if (by_one_n > 0) {
          if (lane < by_one_n) buf[by_one_at + lane] = by_one[lane];
          __syncwarp();
        }
        if (lane == 0) {
          // the copies first; the phase completes with the arrival below
          if (copy_bytes + lone_bytes > 0) mbar_expect_tx(&full_bar[b], copy_bytes + lone_bytes);
          for (uint32_t off = 0; off < copy_bytes; off += kBulkChunk)
            bulk_g2s(reinterpret_cast<char*>(buf) + off, reinterpret_cast<const char*>(src) + off,
                     min(kBulkChunk, copy_bytes - off), &full_bar[b]);
          if (lone_bulk[0]) bulk_g2s(buf + edge0, lone[0], 16u, &full_bar[b]);
          if (lone_bulk[1]) bulk_g2s(buf + edge0 + EPV, lone[1], 16u, &full_bar[b]);
          meta[it % (2 * NB)] = m;
          mbar_arrive(&full_bar[b]);
        }
        ++it;
      }
      if (has_next && nb <= 1) load_dependent(nxt);
      cur = nxt;
    }
    if (!failed) {
      // end of stream
      const int b = it % NB;
      const uint32_t use = it / NB;
      if (use > 0 && !mbar_wait_bounded(&empty_bar[b], (use - 1) & 1)) {
        if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
      } else if (lane == 0) {
        meta[it % (2 * NB)].r = -1;
        mbar_arrive(&full_bar[b]);
      }
    }
    if (lane == 0 && stored) bulk_wait_read_all();
  } else {
    // =============================================================== consumer warps
    // the cluster's loss contributions, added in the order of its rows (rank 0, warp 0, lane 0
    // keeps the sum; one partial per cluster goes to the workspace at the end)
    double cl_loss = 0.0;
    for (uint32_t it = 0;; ++it) {
      const int b = it % NB;
      if (!mbar_wait_bounded(&full_bar[b], (it / NB) & 1)) {
        if (tid == 0) flag_status(p.status, RL_DEV_TIMEOUT);
        break;
      }
      const RowMeta& m = meta[it % (2 * NB)];
      if (m.r < 0) break;
      const int64_t r = m.r;
      const T* buf = buf_base + b * p.buf_elems;
      const int nv = kBlocks ? m.nv : n32 / EPV;
      const int e_n = kBlocks ? m.e_n : n32 % EPV;

      // ---- pass 1: online softmax partial over the slice, which moves into registers here (vector
      // j = tid + k * NC in hold[k]); the stage is released right after, so the next copy lands
      // while the exchange and pass 2 run.
      SoftmaxPartial ps{RL_NEG_INF, 0.f, 0.f};
      uint4 hold[HOLDV];
      float tail_z = 0.f;
      const uint32_t pad = Vec<T>::kPadWord;
      auto reload = [&](int k) {
        const int j = tid + k * NC;
        if (j >= nv) return make_uint4(pad, pad, pad, pad);
        const uint4* at = reinterpret_cast<const uint4*>(buf) + j;
        if constexpr (SHIFT) {
          const int d = m.shift;
          if (d != 0) {
            const uint4 x = at[0], y = at[1];
            return d == 1 ? make_uint4(x.y, x.z, x.w, y.x) : d == 2 ? make_uint4(x.z, x.w, y.x, y.y)
                                                                    : make_uint4(x.w, y.x, y.y, y.z);
          }
        }
        return at[0];
      };
#pragma unroll
      for (int k = 0; k < HOLDV; ++k) hold[k] = reload(k);
      fold_block<T, ENT>(ps, hold, reload);
      // the elements outside the vectors, one per lane of the first two warps
      if (warp < 2 && e_n != 0) {
        if (lane < (warp == 0 ? e_n & 15 : e_n >> 4)) {
          const float z = Vec<T>::to_f(buf[(warp == 0 ? m.e_at : edge0 + EPV) + lane]);
          tail_z = z;
          if (z != RL_NEG_INF) {
            raise_max<ENT>(ps, z);
            accumulate<ENT>(ps, z, -ps.m * kLog2e);
          }
        }
      }
      ps = merge_lanes<T, ENT>(ps);  // the same in every lane
      // warp 0 of the CTA holding the sampled token carries z_a; every other partial carries 0
      const float za_part = (warp == 0 && m.a_at >= 0) ? Vec<T>::to_f(buf[m.a_at]) : 0.f;
      __syncwarp();  // every read of the stage is done
      if (lane == 0) mbar_arrive(&empty_bar[b]);

      // ---- exchange: every warp's partial to every CTA of the cluster (a CTA on its own: to its
      // own mailbox by a plain store and an arrival, without the trip through the cluster's network)
      const int par = it & 1;
      if (C == 1) {
        if (lane == 0) {
          mbox[par][warp] = make_float4(ps.m, ps.s, ps.u, za_part);
          mbar_arrive(&xbar[par]);
        }
      } else {
        if (warp == 0 && lane == 0) mbar_arrive_expect_tx(&xbar[par], C * NW * 16u);
        if (lane < static_cast<int>(C)) {
          const uint32_t dst = map_to_rank(smem_addr(&mbox[par][rank * NW + warp]), lane);
          const uint32_t bar = map_to_rank(smem_addr(&xbar[par]), lane);
          st_async_f4(dst, make_float4(ps.m, ps.s, ps.u, za_part), bar);
        }
      }
      if (!mbar_wait_cluster_bounded(&xbar[par], (it >> 1) & 1)) {
        if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
        break;
      }
      // ---- merge all C * NW partials in a fixed order
      // (lane l takes partials l, l + 32, ...; those with nothing seen, s = 0, do not count)
      const int total = static_cast<int>(C) * NW;
      float4 w0 = make_float4(RL_NEG_INF, 0.f, 0.f, 0.f), w1 = w0;
      if (lane < total) w0 = mbox[par][lane];
      if (lane + 32 < total) w1 = mbox[par][lane + 32];
      SoftmaxPartial q{w0.x, w0.y, w0.z};
      float zsum = w0.w + w1.w;
      if (total > 32) q = merge(q, SoftmaxPartial{w1.x, w1.y, w1.z});
      for (int k = lane + 64; k < total; k += 32) {
        const float4 w = mbox[par][k];
        q = merge(q, SoftmaxPartial{w.x, w.y, w.z});
        zsum += w.w;
      }
      q = merge_lanes<T, ENT>(q);  // the same in every lane
      const float za = warp_sum(zsum);
      const RowLse rl = row_lse<kSplit>(q);
      const float lnS = rl.lnS, lse = rl.hi;
      const float H = ENT ? lnS - q.u / q.s : lnS;  // without the entropy: times 0, for its NaN

      {
        // per-token scalars (every lane computes the same values)
        const float A = m.A, c = m.c, old = m.old;
        const float logp = (za - lse) - rl.lo;
        const float rho = expf(log_ratio<kSplit>(za, old, rl));
        const float crho = fminf(fmaxf(rho, p.clip_lo), p.clip_hi);
        const float surr = fminf(rho * A, crho * A);
        const bool cut = (A > 0.f && rho > p.clip_hi) || (A < 0.f && rho < p.clip_lo);
        const float w = (p.tis_cap > 0.f && p.rollout_logp) ? fminf(expf(old - m.roll), p.tis_cap) : 1.f;
        float kl = 0.f, dkl = 0.f;
        if (p.beta != 0.f && p.ref_logp) {
          const float d = ((m.ref - za) + lse) + rl.lo;  // r - logp
          const float ed = expf(d);
          kl = ed - d - 1.f;
          dkl = 1.f - ed;
        }
        // alpha H also without the bonus (alpha = 0): fminf drops the ratio's NaN, but 0 x ln S is NaN for
        // a row whose softmax is undefined, which has to make the loss NaN
        const float ell = -w * surr + p.beta * kl - p.alpha * H;
        const float g = (cut ? 0.f : -w * A * rho) + p.beta * dkl;
        const float cg = c * g, ca0 = c * p.alpha;
        // p_v = 2^(z_v log2(e) + nl) with nl = fl(-lse log2(e)); its rounding scales every p_v of
        // the row by 2^errl (errl exact by one fma), folded into the coefficients below
        const float nl = -lse * kLog2e;
        const float fl = fmaf(fmaf(-lse, kLog2e, -nl), kLn2, 1.f - rl.lo);
        const float Kp = -cg * fl;                      // gradient = Kp p_v (+ cg at v = a)
        const float ca = ca0 * fl;                      // entropy: p_v (ca z_v + Ke)
        const float Ke = (-cg + ca0 * (H - lse)) * fl;
        if (rank == 0 && warp == 0 && lane == 0) {
          cl_loss += static_cast<double>(c) * static_cast<double>(ell);
          if (p.token_stats) {
            float* st = p.token_stats + r * 5;
            st[0] = logp; st[1] = rho; st[2] = cut ? 1.f : 0.f; st[3] = H; st[4] = kl;
          }
        }
        // ---- pass 2: gradient from the on-chip slice
        T* g_vec = grad + (kBlocks ? m.base : r * ld + s0 * EPV);
        auto grad_of = [&](float z) {
          const float pk = ex2(fmaf(z, kLog2e, nl));
          return ENT ? pk * fmaf(ca, fmaxf(z, -1e30f), Ke) : Kp * pk;
        };
        constexpr int NP = Vec<T>::NP;
        const float2 l2 = make_float2(kLog2e, kLog2e), nl2 = make_float2(nl, nl);
        const float2 kp2 = make_float2(Kp, Kp), ca2 = make_float2(ca, ca), ke2 = make_float2(Ke, Ke);
#pragma unroll
        for (int k = 0; k < HOLDV; ++k) {
          const int j = tid + k * NC;
          float2 q[NP], o[NP];
          Vec<T>::pairs(hold[k], q);
#pragma unroll
          for (int i = 0; i < NP; ++i) {
            const float2 xx = __ffma2_rn(q[i], l2, nl2);
            const float2 pk = make_float2(ex2(xx.x), ex2(xx.y));
            if (ENT) {
              const float2 zc = make_float2(fmaxf(q[i].x, -1e30f), fmaxf(q[i].y, -1e30f));
              o[i] = __fmul2_rn(pk, __ffma2_rn(ca2, zc, ke2));
            } else {
              o[i] = __fmul2_rn(kp2, pk);
            }
          }
          if constexpr (SHIFT) {
            // fp32 vectors that start d elements into a block: the block from this lane's element
            // h = 4 - d on ends with the next lane's first h
            const int d = m.shift, h = EPV - d;
            const float o0 = o[0].x, o1 = o[0].y, o2 = o[1].x, o3 = o[1].y;
            const float n0 = __shfl_down_sync(0xffffffffu, o0, 1), n1 = __shfl_down_sync(0xffffffffu, o1, 1),
                        n2 = __shfl_down_sync(0xffffffffu, o2, 1);
            float* g = reinterpret_cast<float*>(g_vec) + j * EPV;
            if (j < nv) {
              if (d == 0) {
                *reinterpret_cast<float4*>(g) = make_float4(o0, o1, o2, o3);
              } else {
                if (lane < 31 && j + 1 < nv) {
                  *reinterpret_cast<float4*>(g + h) = h == 1   ? make_float4(o1, o2, o3, n0)
                                                      : h == 2 ? make_float4(o2, o3, n0, n1)
                                                               : make_float4(o3, n0, n1, n2);
                } else {
                  if (h <= 1) g[1] = o1;
                  if (h <= 2) g[2] = o2;
                  g[3] = o3;
                }
                if (lane == 0) {
                  g[0] = o0;
                  if (h >= 2) g[1] = o1;
                  if (h >= 3) g[2] = o2;
                }
              }
            }
          } else {
            if (j < nv) st_global_16(g_vec + j * EPV, Vec<T>::pack_pairs(o));
          }
        }
        if (warp < 2 && e_n != 0 && lane < (warp == 0 ? e_n & 15 : e_n >> 4))
          Vec<T>::store_scalar(g_vec + (warp == 0 && kBlocks ? m.e_rel : nv * EPV) + lane, grad_of(tail_z));
        // the sampled token's element gets + c g; rewritten by the thread that stored it
        if (tid == m.a_writer) Vec<T>::store_scalar(g_vec + m.a_rel, grad_of(za) + cg);
      }
    }
    if (rank == 0 && warp == 0) {
      // one partial per cluster (cid < clusters <= rows); the last cluster to finish adds all
      // of them, in a fixed order, into the caller's total, so no second launch is needed
      __syncwarp();
      uint32_t last = 0;
      if (lane == 0) {
        p.row_loss[cid] = cl_loss;
        __threadfence();
        last = atomicAdd(p.done, 1u) == static_cast<uint32_t>(ncl - 1) ? 1u : 0u;
        if (last) __threadfence();
      }
      __syncwarp();
      last = __shfl_sync(0xffffffffu, last, 0);
      if (last) {
        double t = 0.0;
        for (int64_t k = lane; k < ncl; k += 32) t += __ldcg(p.row_loss + k);
        t = warp_sum(t);
        if (lane == 0) {
          *p.loss_accum += t;
          *p.done = 0u;
        }
      }
    }
  }
  __syncthreads();
  // no CTA leaves while a peer may still write into its mailbox
  if (C > 1) cluster_sync_all();
}

// ------------------------------------------------------------------ fp32 rows on 16-byte boundaries
//
// fp32 rows of up to 129,024 entries whose leading dimension is a multiple of four keep a kernel of
// their own: the same split as rows_kernel's fp32 form and the same bits (the order of the sums is
// part of the fp32 path's results, see merge_lanes), with a row's words held by each consumer and its
// places worked out there. A stage is released only once the row's exchange has arrived. On the edge
// batch (32,768 rows of 32,000 entries, 38% of them zero-filled; HBM's floor 1,008 us) that takes 1,066 us, an
// early release 1,102 to 1,147 us, and rows_kernel on the same shape 1,136 us either way. How the compiler
// allots the consumers' registers moves this kernel by 5%, by V in either direction (a build without its
// 4 bytes of spills 1,140 us there, but 6% faster at 80,000 entries); why is not known. Fewer clusters than
// fit, a release after the gradient's stores: slower.
// Slices of at most 30 KB (clusters of 5 at V = 32,000), 7 consumer warps of up to 9
// vectors, 3 CTAs per SM: 4.15 ms per 131,072 rows against 4.35 with clusters of 4 at 2 per SM.
constexpr int kF32Warps = 7, kF32Hold = 9;

struct F32Meta {
  int64_t r;  // row index, -1 = end of the stream
  int32_t a;  // sampled token id
  float A, c, old, ref, roll;
};

template <bool ENT>
__global__ void __launch_bounds__((kF32Warps + 1) * 32, 3) rows_f32_kernel(const RowArgs p) {
  using T = float;
  constexpr int NW = kF32Warps, HOLDV = kF32Hold, kZeroBytes = 2048;
  constexpr int EPV = Vec<T>::N;
  constexpr int NB = RL_STAGES;
  constexpr int NC = NW * 32;  // consumer threads
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[NB], empty_bar[NB], xbar[2];
  __shared__ F32Meta meta[NB];
  __shared__ __align__(16) float4 mbox[2][kMaxCluster * NW];
  __shared__ __align__(128) uint4 zeros[kZeroBytes / 16];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = cluster_ctarank(), C = cluster_nctarank();
  const int64_t cid = blockIdx.x / C, ncl = gridDim.x / C;
  const int64_t rows = p.rows, V = p.V, ld = p.ld;
  const int64_t s0 = static_cast<int64_t>(rank) * p.slice;
  const int64_t n_end = (s0 + p.slice < V) ? s0 + p.slice : V;
  const int n = n_end > s0 ? static_cast<int>(n_end - s0) : 0;  // elements of my slice
  const int nv = n / EPV;                                        // full 16-byte vectors
  const uint32_t tma_bytes = static_cast<uint32_t>(nv * 16);
  const T* logits = static_cast<const T*>(p.logits);
  T* grad = static_cast<T*>(p.grad);
  T* const buf_base = reinterpret_cast<T*>(smem_raw);

  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < NB; ++k) {
      mbar_init(&full_bar[k], 1);
      mbar_init(&empty_bar[k], NW);
    }
    mbar_init(&xbar[0], C == 1 ? NW : 1);
    mbar_init(&xbar[1], C == 1 ? NW : 1);
    fence_mbar_init();
  }
  for (int k = tid; k < kZeroBytes / 16; k += blockDim.x) zeros[k] = make_uint4(0, 0, 0, 0);
  fence_proxy_async_smem();
  __syncthreads();
  if (C > 1) cluster_sync_all();  // every peer's mailbox barrier exists before the first st.async

  if (warp == NW) {
    // =============================================================== producer warp
    // Row metadata is fetched 32 rows at a time, one row per lane, and handed row by row to the
    // staging loop with shuffles. The loads of the next batch are issued while the current one
    // is staged (its owners' coefficients once the owners have arrived), so their latency is
    // hidden behind the copies.
    uint32_t it = 0;
    bool failed = false, stored = false;
    struct Batch {
      int32_t a, i;
      uint32_t m;
      float c, A, old, ref, roll;
    };
    auto load_primary = [&](int64_t b0, Batch& q) {
      const int64_t my = b0 + static_cast<int64_t>(lane) * ncl;
      q = Batch{0, -1, 0u, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (my < rows) {
        q.a = p.token_ids[my];
        q.m = p.mask[my];
        q.i = p.token_traj[my];
        q.old = p.old_logp[my];
        if (p.ref_logp) q.ref = p.ref_logp[my];
        if (p.rollout_logp) q.roll = p.rollout_logp[my];
        if (p.adv_per_row) q.A = p.adv[my];
      }
    };
    auto load_dependent = [&](Batch& q) {
      if (q.m != 0 && q.i >= 0 && q.i < p.n_traj) {
        q.c = p.coef[q.i];
        if (!p.adv_per_row) q.A = p.adv[q.i];
      }
    };
    Batch cur, nxt = Batch{0, -1, 0u, 0.f, 0.f, 0.f, 0.f, 0.f};
    load_primary(cid, cur);
    load_dependent(cur);
    for (int64_t base = cid; base < rows && !failed; base += 32 * ncl) {
      const int64_t next_base = base + 32 * ncl;
      const bool has_next = next_base < rows;
      if (has_next) load_primary(next_base, nxt);
      const int32_t la = cur.a, li = cur.i;
      const uint32_t lm = cur.m;
      const float lc = cur.c, lA = cur.A, lold = cur.old, lref = cur.ref, lroll = cur.roll;
      const int nb = static_cast<int>(min(static_cast<int64_t>(32), (rows - base + ncl - 1) / ncl));
      for (int jr = 0; jr < nb && !failed; ++jr) {
        if (jr == 1 && has_next) load_dependent(nxt);  // the next batch's owners have arrived by now
        const int64_t r = base + static_cast<int64_t>(jr) * ncl;
        F32Meta m;
        bool active = true;
        m.r = r;
        m.a = __shfl_sync(0xffffffffu, la, jr);
        active = __shfl_sync(0xffffffffu, lm, jr) != 0;
        if (active) {
          const int32_t i = __shfl_sync(0xffffffffu, li, jr);
          if (i < 0 || i >= p.n_traj) {
            if (rank == 0 && lane == 0) flag_status(p.status, RL_DEV_BAD_TRAJ);
            active = false;
          } else {
            m.c = __shfl_sync(0xffffffffu, lc, jr);
            m.A = __shfl_sync(0xffffffffu, lA, jr);
            active = m.c != 0.f;
            if (active && (m.a < 0 || m.a >= V)) {
              if (rank == 0 && lane == 0) flag_status(p.status, RL_DEV_BAD_TOKEN);
              active = false;
            }
          }
        }
        if (!active) {
          // zero this CTA's slice of gradient row r
          T* g = grad + r * ld + s0;
          if (lane == 0) {
            const uint32_t bytes = tma_bytes;
            for (uint32_t off = 0; off < bytes; off += kZeroBytes)
              bulk_s2g(reinterpret_cast<char*>(g) + off, zeros, min(static_cast<uint32_t>(kZeroBytes), bytes - off));
            bulk_commit();
            stored = true;
          }
          for (int e = nv * EPV + lane; e < n; e += 32) g[e] = T(0);
          if (rank == 0 && lane == 0 && p.token_stats)
            for (int k = 0; k < 5; ++k) p.token_stats[r * 5 + k] = 0.f;
          continue;
        }
        m.old = __shfl_sync(0xffffffffu, lold, jr);
        m.ref = __shfl_sync(0xffffffffu, lref, jr);
        m.roll = __shfl_sync(0xffffffffu, lroll, jr);
        const int b = it % NB;
        const uint32_t use = it / NB;
        if (use > 0 && !mbar_wait_bounded(&empty_bar[b], (use - 1) & 1)) {
          failed = true;
          if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
          break;
        }
        T* buf = buf_base + b * p.buf_elems;
        const T* src = logits + r * ld + s0;
        for (int e = nv * EPV + lane; e < n; e += 32) buf[e] = src[e];
        __syncwarp();
        if (lane == 0) {
          meta[b] = m;
          if (tma_bytes > 0) {
            mbar_arrive_expect_tx(&full_bar[b], tma_bytes);
            for (uint32_t off = 0; off < tma_bytes; off += kBulkChunk)
              bulk_g2s(reinterpret_cast<char*>(buf) + off, reinterpret_cast<const char*>(src) + off,
                       min(kBulkChunk, tma_bytes - off), &full_bar[b]);
          } else {
            mbar_arrive(&full_bar[b]);
          }
        }
        ++it;
      }
      if (has_next && nb <= 1) load_dependent(nxt);
      cur = nxt;
    }
    if (!failed) {
      // end of stream
      const int b = it % NB;
      const uint32_t use = it / NB;
      if (use > 0 && !mbar_wait_bounded(&empty_bar[b], (use - 1) & 1)) {
        if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
      } else if (lane == 0) {
        meta[b].r = -1;
        mbar_arrive(&full_bar[b]);
      }
    }
    if (lane == 0 && stored) bulk_wait_read_all();
  } else {
    // =============================================================== consumer warps
    // the cluster's loss contributions, added in the order of its rows (rank 0, warp 0, lane 0
    // keeps the sum; one partial per cluster goes to the workspace at the end)
    double cl_loss = 0.0;
    for (uint32_t it = 0;; ++it) {
      const int b = it % NB;
      if (!mbar_wait_bounded(&full_bar[b], (it / NB) & 1)) {
        if (tid == 0) flag_status(p.status, RL_DEV_TIMEOUT);
        break;
      }
      const F32Meta m = meta[b];
      if (m.r < 0) break;
      const int64_t r = m.r;
      const T* buf = buf_base + b * p.buf_elems;
      const int32_t a = m.a;
      const bool a_ok = a >= 0 && a < V;
      const uint32_t owner = a_ok ? static_cast<uint32_t>(a / p.slice) : 0u;

      // ---- pass 1: online softmax partial over the slice, which moves into registers here (vector
      // j = tid + k * NC in hold[k]); the stage is released after the exchange (above).
      SoftmaxPartial ps{RL_NEG_INF, 0.f, 0.f};
      uint4 hold[HOLDV];
      float tail_z = 0.f;
      const uint32_t pad = Vec<T>::kPadWord;
      auto reload = [&](int k) {
        const int j = tid + k * NC;
        return j < nv ? reinterpret_cast<const uint4*>(buf)[j] : make_uint4(pad, pad, pad, pad);
      };
#pragma unroll
      for (int k = 0; k < HOLDV; ++k) hold[k] = reload(k);
      fold_block<T, ENT>(ps, hold, reload);
      // ragged tail (fewer than EPV elements): one per thread at most
      if (nv * EPV + tid < n) {
        const float z = Vec<T>::to_f(buf[nv * EPV + tid]);
        tail_z = z;
        if (z != RL_NEG_INF) {
          raise_max<ENT>(ps, z);
          accumulate<ENT>(ps, z, -ps.m * kLog2e);
        }
      }
      ps = merge_lanes<T, ENT>(ps);  // the same in every lane
      // warp 0 of the CTA holding the sampled token carries z_a; every other partial carries 0
      const float za_part = (warp == 0 && a_ok && rank == owner) ? Vec<T>::to_f(buf[a - s0]) : 0.f;

      // ---- exchange: every warp's partial to every CTA of the cluster (a CTA on its own: to its
      // own mailbox by a plain store and an arrival, without the trip through the cluster's network)
      const int par = it & 1;
      if (C == 1) {
        if (lane == 0) {
          mbox[par][warp] = make_float4(ps.m, ps.s, ps.u, za_part);
          mbar_arrive(&xbar[par]);
        }
      } else {
        if (warp == 0 && lane == 0) mbar_arrive_expect_tx(&xbar[par], C * NW * 16u);
        if (lane < static_cast<int>(C)) {
          const uint32_t dst = map_to_rank(smem_addr(&mbox[par][rank * NW + warp]), lane);
          const uint32_t bar = map_to_rank(smem_addr(&xbar[par]), lane);
          st_async_f4(dst, make_float4(ps.m, ps.s, ps.u, za_part), bar);
        }
      }
      if (!mbar_wait_cluster_bounded(&xbar[par], (it >> 1) & 1)) {
        if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
        break;
      }
      __syncwarp();  // every read of the stage is done
      if (lane == 0) mbar_arrive(&empty_bar[b]);
      // ---- merge all C * NW partials in a fixed order
      // (lane l takes partials l, l + 32, ...; those with nothing seen, s = 0, do not count)
      const int total = static_cast<int>(C) * NW;
      float4 w0 = make_float4(RL_NEG_INF, 0.f, 0.f, 0.f), w1 = w0;
      if (lane < total) w0 = mbox[par][lane];
      if (lane + 32 < total) w1 = mbox[par][lane + 32];
      SoftmaxPartial q{w0.x, w0.y, w0.z};
      float zsum = w0.w + w1.w;
      if (total > 32) q = merge(q, SoftmaxPartial{w1.x, w1.y, w1.z});
      for (int k = lane + 64; k < total; k += 32) {
        const float4 w = mbox[par][k];
        q = merge(q, SoftmaxPartial{w.x, w.y, w.z});
        zsum += w.w;
      }
      q = merge_lanes<T, ENT>(q);  // the same in every lane
      const float za = warp_sum(zsum);
      const RowLse rl = row_lse<false>(q);
      const float lnS = rl.lnS, lse = rl.hi;
      const float H = lnS - q.u / q.s;  // without the entropy: times 0, for its NaN

      {
        // per-token scalars (every lane computes the same values)
        const float A = m.A, c = m.c, old = m.old;
        const float logp = (za - lse) - rl.lo;
        const float rho = expf(log_ratio<false>(za, old, rl));
        const float crho = fminf(fmaxf(rho, p.clip_lo), p.clip_hi);
        const float surr = fminf(rho * A, crho * A);
        const bool cut = (A > 0.f && rho > p.clip_hi) || (A < 0.f && rho < p.clip_lo);
        const float w = (p.tis_cap > 0.f && p.rollout_logp) ? fminf(expf(old - m.roll), p.tis_cap) : 1.f;
        float kl = 0.f, dkl = 0.f;
        if (p.beta != 0.f && p.ref_logp) {
          const float d = ((m.ref - za) + lse) + rl.lo;  // r - logp
          const float ed = expf(d);
          kl = ed - d - 1.f;
          dkl = 1.f - ed;
        }
        const float ell = -w * surr + p.beta * kl - p.alpha * H;
        const float g = (cut ? 0.f : -w * A * rho) + p.beta * dkl;
        const float cg = c * g, ca0 = c * p.alpha;
        // p_v = 2^(z_v log2(e) + nl) with nl = fl(-lse log2(e)); its rounding scales every p_v of
        // the row by 2^errl (errl exact by one fma), folded into the coefficients below
        const float nl = -lse * kLog2e;
        const float fl = fmaf(fmaf(-lse, kLog2e, -nl), kLn2, 1.f - rl.lo);
        const float Kp = -cg * fl;                      // gradient = Kp p_v (+ cg at v = a)
        const float ca = ca0 * fl;                      // entropy: p_v (ca z_v + Ke)
        const float Ke = (-cg + ca0 * (H - lse)) * fl;
        if (rank == 0 && warp == 0 && lane == 0) {
          cl_loss += static_cast<double>(c) * static_cast<double>(ell);
          if (p.token_stats) {
            float* st = p.token_stats + r * 5;
            st[0] = logp; st[1] = rho; st[2] = cut ? 1.f : 0.f; st[3] = H; st[4] = kl;
          }
        }
        // ---- pass 2: gradient from the on-chip slice
        T* g_row = grad + r * ld + s0;
        {
          constexpr int NP = Vec<T>::NP;
          const float2 l2 = make_float2(kLog2e, kLog2e), nl2 = make_float2(nl, nl);
          const float2 kp2 = make_float2(Kp, Kp), ca2 = make_float2(ca, ca), ke2 = make_float2(Ke, Ke);
#pragma unroll
          for (int k = 0; k < HOLDV; ++k) {
            const int j = tid + k * NC;
            float2 q[NP], o[NP];
            Vec<T>::pairs(hold[k], q);
#pragma unroll
            for (int i = 0; i < NP; ++i) {
              const float2 xx = __ffma2_rn(q[i], l2, nl2);
              const float2 pk = make_float2(ex2(xx.x), ex2(xx.y));
              if (ENT) {
                const float2 zc = make_float2(fmaxf(q[i].x, -1e30f), fmaxf(q[i].y, -1e30f));
                o[i] = __fmul2_rn(pk, __ffma2_rn(ca2, zc, ke2));
              } else {
                o[i] = __fmul2_rn(kp2, pk);
              }
            }
            if (j < nv) st_global_16(g_row + j * EPV, Vec<T>::pack_pairs(o));
          }
        }
        if (nv * EPV + tid < n) {
          const float z = tail_z;
          const float pk = ex2(fmaf(z, kLog2e, nl));
          Vec<T>::store_scalar(g_row + nv * EPV + tid, ENT ? pk * fmaf(ca, fmaxf(z, -1e30f), Ke) : Kp * pk);
        }
        // the sampled token's element gets + c g; rewritten by the thread that stored it
        if (rank == owner) {
          const int ia = static_cast<int>(a - s0);
          const int writer = ia < nv * EPV ? (ia / EPV) % NC : (ia - nv * EPV);
          if (tid == writer) {
            const float pk = ex2(fmaf(za, kLog2e, nl));
            const float ga = (ENT ? pk * fmaf(ca, fmaxf(za, -1e30f), Ke) : Kp * pk) + cg;
            Vec<T>::store_scalar(g_row + ia, ga);
          }
        }
      }
    }
    if (rank == 0 && warp == 0) {
      // one partial per cluster (cid < clusters <= rows); the last cluster to finish adds all
      // of them, in a fixed order, into the caller's total, so no second launch is needed
      __syncwarp();
      uint32_t last = 0;
      if (lane == 0) {
        p.row_loss[cid] = cl_loss;
        __threadfence();
        last = atomicAdd(p.done, 1u) == static_cast<uint32_t>(ncl - 1) ? 1u : 0u;
        if (last) __threadfence();
      }
      __syncwarp();
      last = __shfl_sync(0xffffffffu, last, 0);
      if (last) {
        double t = 0.0;
        for (int64_t k = lane; k < ncl; k += 32) t += __ldcg(p.row_loss + k);
        t = warp_sum(t);
        if (lane == 0) {
          *p.loss_accum += t;
          *p.done = 0u;
        }
      }
    }
  }
  __syncthreads();
  // no CTA leaves while a peer may still write into its mailbox
  if (C > 1) cluster_sync_all();
}

// ------------------------------------------------------------------ short rows
//
// For rows of at most kSmallRowBytes (V <= 4,096 bf16 or 2,048 fp32) a cluster of CTAs per row, or
// a CTA that streams it, costs more in set-up, barriers and exchange than the row's own data. Here
// one warp owns a row: its lanes hold the row's whole blocks in registers (block j = lane + 32 k in
// x[k]; NV of them, the smallest of 4, 8 and 16 that holds the row, so that a short row neither
// computes on pads nor keeps other warps off the SM), the elements of the partial blocks at its
// ends one per lane, fold them with the same online softmax as the cluster kernel, merge the 32
// partials by shuffles, and write the gradient from registers. Warps take rows w, w + (all warps),
// ..., with the next row's words fetched a row ahead; each warp adds its rows' loss terms in row
// order, the CTA adds its warps' sums in warp order into one partial, and the last CTA to finish
// (the same workspace counter as the cluster kernel's) adds the CTAs' partials, in order, into
// the caller's total.
constexpr int64_t kSmallRowBytes = 8192;
constexpr int kSmallWarps = 8;

// CTAs per SM the registers are budgeted for, by the blocks a lane holds: as many as leave no
// spills.
template <typename T, int NV>
constexpr int small_ctas(bool loss) {
  if (!loss) return NV == 16 ? 2 : NV == 8 ? 3 : 4;
  return NV == 16 || (NV == 8 && sizeof(T) == 4) ? 2 : 3;
}

// A lane's part of a short row: its whole blocks, and at most one element of the partial blocks
// (the head's by lanes 0-7, the tail's by lanes 8-15).
template <typename T, int NV>
struct SmallRow {
  static constexpr int EPV = Vec<T>::N;
  const T* row;
  RowSpan<T> span;
  int edge;  // element of the row, -1: none
  uint4 x[NV];
  float ez;  // its value
  __device__ __forceinline__ void locate(const T* logits, int64_t r, int64_t ld, int64_t V, int lane) {
    row = logits + r * ld;
    span = row_span<T>(r, ld, V);
    edge = lane < span.head ? lane
           : lane >= 8 && lane - 8 < span.tail ? static_cast<int>(V) - span.tail + lane - 8 : -1;
  }
  int b0;    // first block of the part that is loaded (long rows go part by part)
  __device__ __forceinline__ uint4 block(int k, int lane) const {
    const int j = b0 + lane + k * 32;
    const uint32_t pad = Vec<T>::kPadWord;
    return j < span.vecs ? reinterpret_cast<const uint4*>(row + span.head)[j] : make_uint4(pad, pad, pad, pad);
  }
  __device__ __forceinline__ void load(int lane, int first = 0) {
    b0 = first;
#pragma unroll
    for (int k = 0; k < NV; ++k) x[k] = block(k, lane);
    ez = edge >= 0 ? Vec<T>::to_f(row[edge]) : 0.f;
  }
  // the warp's partial, the same in every lane
  template <bool ENT>
  __device__ __forceinline__ SoftmaxPartial fold(int lane) {
    SoftmaxPartial ps{RL_NEG_INF, 0.f, 0.f};
    fold_part<ENT>(ps, lane);
    return finish<ENT>(ps, ps.s == 0.f, lane);
  }
  template <bool ENT>
  __device__ __forceinline__ void fold_part(SoftmaxPartial& ps, int lane) {
    fold_block<T, ENT, NV, false>(ps, x, [&](int k) { return block(k, lane); });
  }
  // A lane that had seen nothing after some part (`none`) had only -inf or NaNs there, which no maximum
  // sees: looked for here, where the row's words are no longer held (kept as references, as the cluster
  // kernels do, they cost 5 to 7% of the forward call at 4,096 and 5,000 entries).
  template <bool ENT>
  __device__ __forceinline__ SoftmaxPartial finish(SoftmaxPartial ps, bool none, int lane) {
    if (none) {
      for (int j = lane; j < span.vecs; j += 32) {
        float2 q[Vec<T>::NP];
        Vec<T>::pairs(reinterpret_cast<const uint4*>(row + span.head)[j], q);
        for (int i = 0; i < Vec<T>::NP; ++i)
          if (q[i].x != q[i].x || q[i].y != q[i].y) ps.s = __int_as_float(0x7fffffff);
      }
    }
    if (edge >= 0 && ez != RL_NEG_INF) {
      raise_max<ENT>(ps, ez);
      accumulate<ENT>(ps, ez, -ps.m * kLog2e);
    }
    return merge_lanes<T, ENT>(ps);
  }
};

template <typename T, bool ENT, int NV>
__global__ void __launch_bounds__(kSmallWarps * 32, small_ctas<T, NV>(true)) small_rows_kernel(const RowArgs p) {
  constexpr bool kSplit = sizeof(T) == 2;
  constexpr int EPV = Vec<T>::N;
  __shared__ double warp_loss[kSmallWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t all_warps = static_cast<int64_t>(gridDim.x) * kSmallWarps;
  const int64_t V = p.V, ld = p.ld;
  const T* logits = static_cast<const T*>(p.logits);
  T* grad = static_cast<T*>(p.grad);
  double w_loss = 0.0;  // lane 0: this warp's rows' c l, in row order
  // A row's own words, fetched a row ahead; its owner's coefficient and advantage are fetched
  // together with the row's logits (when the row is masked in and its owner in range), so that a
  // row costs one dependent trip to memory before its arithmetic, two for a warp's first row.
  struct Words {
    int32_t a, i;
    uint32_t mk;
    float old, ref, roll, A;
  };
  auto fetch_words = [&](int64_t r) {
    Words w = {0, -1, 0u, 0.f, 0.f, 0.f, 0.f};
    if (r < p.rows) {
      w.a = p.token_ids[r];
      w.mk = p.mask[r];
      w.i = p.token_traj[r];
      w.old = p.old_logp[r];
      if (p.ref_logp) w.ref = p.ref_logp[r];
      if (p.rollout_logp) w.roll = p.rollout_logp[r];
      if (p.adv_per_row) w.A = p.adv[r];
    }
    return w;
  };
  int64_t r = static_cast<int64_t>(blockIdx.x) * kSmallWarps + warp;
  Words next = fetch_words(r);
  for (; r < p.rows; r += all_warps) {
    const Words wd = next;
    // ---- which rows are trained on (the same tests, in the same order, as the cluster kernel)
    const int32_t a = wd.a, i = wd.i;
    const bool owner_ok = i >= 0 && i < p.n_traj;
    const bool fetch = wd.mk != 0 && owner_ok;
    SmallRow<T, NV> sr;
    sr.locate(logits, r, ld, V, lane);
    float c = 0.f, A = 0.f, za = 0.f;
    if (fetch) {
      c = p.coef[i];
      A = p.adv_per_row ? wd.A : p.adv[i];
      if (a >= 0 && a < V) za = Vec<T>::to_f(sr.row[a]);
      sr.load(lane);
    }
    next = fetch_words(r + all_warps);
    bool active = fetch && c != 0.f;
    if (wd.mk != 0 && !owner_ok && lane == 0) flag_status(p.status, RL_DEV_BAD_TRAJ);
    if (active && (a < 0 || a >= V)) {
      if (lane == 0) flag_status(p.status, RL_DEV_BAD_TOKEN);
      active = false;
    }
    T* g_row = grad + r * ld;
    T* g_vec = g_row + sr.span.head;
    if (!active) {
      for (int j = lane; j < sr.span.vecs; j += 32) st_global_16(g_vec + j * EPV, make_uint4(0u, 0u, 0u, 0u));
      if (sr.edge >= 0) g_row[sr.edge] = T(0);
      if (lane == 0 && p.token_stats)
        for (int k = 0; k < 5; ++k) p.token_stats[r * 5 + k] = 0.f;
      continue;
    }
    // ---- pass 1
    const SoftmaxPartial q = sr.template fold<ENT>(lane);
    const RowLse rl = row_lse<kSplit>(q);
    const float lnS = rl.lnS, lse = rl.hi;
    const float H = ENT ? lnS - q.u / q.s : lnS;  // without the entropy: times 0, for its NaN
    // ---- per-token scalars (every lane computes the same values)
    const float old = wd.old;
    const float logp = (za - lse) - rl.lo;
    const float rho = expf(log_ratio<kSplit>(za, old, rl));
    const float crho = fminf(fmaxf(rho, p.clip_lo), p.clip_hi);
    const float surr = fminf(rho * A, crho * A);
    const bool cut = (A > 0.f && rho > p.clip_hi) || (A < 0.f && rho < p.clip_lo);
    const float w = (p.tis_cap > 0.f && p.rollout_logp) ? fminf(expf(old - wd.roll), p.tis_cap) : 1.f;
    float kl = 0.f, dkl = 0.f;
    if (p.beta != 0.f && p.ref_logp) {
      const float d = ((wd.ref - za) + lse) + rl.lo;  // r - logp
      const float ed = expf(d);
      kl = ed - d - 1.f;
      dkl = 1.f - ed;
    }
    const float ell = -w * surr + p.beta * kl - p.alpha * H;
    const float g = (cut ? 0.f : -w * A * rho) + p.beta * dkl;
    const float cg = c * g, ca0 = c * p.alpha;
    // p_v = 2^(z_v log2(e) + nl), the rounding of nl folded into the coefficients (as in the
    // cluster kernel)
    const float nl = -lse * kLog2e;
    const float fl = fmaf(fmaf(-lse, kLog2e, -nl), kLn2, 1.f - rl.lo);
    const float Kp = -cg * fl;
    const float ca = ca0 * fl;
    const float Ke = (-cg + ca0 * (H - lse)) * fl;
    if (lane == 0) {
      w_loss += static_cast<double>(c) * static_cast<double>(ell);
      if (p.token_stats) {
        float* st = p.token_stats + r * 5;
        st[0] = logp; st[1] = rho; st[2] = cut ? 1.f : 0.f; st[3] = H; st[4] = kl;
      }
    }
    __syncwarp();  // every lane has read z_a before any lane overwrites it (in-place gradients)
    // ---- pass 2: gradient from the registers
    constexpr int NP = Vec<T>::NP;
    const float2 l2 = make_float2(kLog2e, kLog2e), nl2 = make_float2(nl, nl);
    const float2 kp2 = make_float2(Kp, Kp), ca2 = make_float2(ca, ca), ke2 = make_float2(Ke, Ke);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int j = lane + k * 32;
      float2 qv[NP], o[NP];
      Vec<T>::pairs(sr.x[k], qv);
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const float2 xx = __ffma2_rn(qv[i], l2, nl2);
        const float2 pk = make_float2(ex2(xx.x), ex2(xx.y));
        if (ENT) {
          const float2 zc = make_float2(fmaxf(qv[i].x, -1e30f), fmaxf(qv[i].y, -1e30f));
          o[i] = __fmul2_rn(pk, __ffma2_rn(ca2, zc, ke2));
        } else {
          o[i] = __fmul2_rn(kp2, pk);
        }
      }
      if (j < sr.span.vecs) st_global_16(g_vec + j * EPV, Vec<T>::pack_pairs(o));
    }
    auto grad_of = [&](float z) {
      const float pk = ex2(fmaf(z, kLog2e, nl));
      return ENT ? pk * fmaf(ca, fmaxf(z, -1e30f), Ke) : Kp * pk;
    };
    if (sr.edge >= 0) Vec<T>::store_scalar(g_row + sr.edge, grad_of(sr.ez));
    // the sampled token's element gets + c g; rewritten by the lane that stored it
    const int tail0 = static_cast<int>(V) - sr.span.tail;
    const int writer = a < sr.span.head ? a : a >= tail0 ? 8 + (a - tail0) : (a - sr.span.head) / EPV % 32;
    if (lane == writer) Vec<T>::store_scalar(g_row + a, grad_of(za) + cg);
  }
  // ---- the loss: warps in order into one partial per CTA; the last CTA adds the partials, all
  // its threads loading them at once (thread k takes partials k, k + 256, ...), then combined
  // by shuffles and the warps in order: a fixed order for a given grid
  __shared__ uint32_t is_last;
  if (lane == 0) warp_loss[warp] = w_loss;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < kSmallWarps; ++k) t += warp_loss[k];
    p.row_loss[blockIdx.x] = t;
    __threadfence();
    is_last = atomicAdd(p.done, 1u) == gridDim.x - 1 ? 1u : 0u;
  }
  __syncthreads();
  if (is_last) {
    __threadfence();
    double t = 0.0;
    for (unsigned k = threadIdx.x; k < gridDim.x; k += kSmallWarps * 32) t += __ldcg(p.row_loss + k);
    t = warp_sum(t);
    if (lane == 0) warp_loss[warp] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int k = 0; k < kSmallWarps; ++k) sum += warp_loss[k];
      *p.loss_accum += sum;
      *p.done = 0u;
    }
  }
}

struct StreamArgs {
  const void* logits;
  int64_t rows, V, ld;
  const int32_t* token_ids;
  float* logp_out;
  float* entropy_out;
  float* lse_out;
  int32_t* status;
  int32_t chunk;      // 16-byte blocks per chunk
  int64_t buf_elems;  // element stride between stages
};

// Forward-only log-probs of short rows: the same warp per row, without a gradient. Rows of more than
// kSmallRowBytes go part by part (NV = 16), up to two parts, or four for bf16 with the entropy, where
// a CTA that streams the row is bound by its row ends and chunk ends. GB/s read, streamed and by
// warps: bf16 V = 1,000 488 and 5,031, 4,096 1,871 and 6,954, 5,000 3,728 and 6,076, 8,192 5,950 and
// 7,001, 16,384 6,889 and 6,738; with the entropy 16,384 5,187 and 6,825; fp32 4,100 4,904 and 6,749.
template <typename T, bool ENT, int NV>
__global__ void __launch_bounds__(kSmallWarps * 32, small_ctas<T, NV>(false)) small_logprobs_kernel(const StreamArgs p) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t all_warps = static_cast<int64_t>(gridDim.x) * kSmallWarps;
  const T* logits = static_cast<const T*>(p.logits);
  int64_t r = static_cast<int64_t>(blockIdx.x) * kSmallWarps + warp;
  int32_t next = r < p.rows ? p.token_ids[r] : 0;
  for (; r < p.rows; r += all_warps) {
    const int32_t a = next;
    const bool a_ok = a >= 0 && a < p.V;
    SmallRow<T, NV> sr;
    sr.locate(logits, r, p.ld, p.V, lane);
    const float za = a_ok ? Vec<T>::to_f(sr.row[a]) : 0.f;
    sr.load(lane);
    next = r + all_warps < p.rows ? p.token_ids[r + all_warps] : 0;
    SoftmaxPartial ps{RL_NEG_INF, 0.f, 0.f};
    sr.template fold_part<ENT>(ps, lane);
    bool none = ps.s == 0.f;
    if (NV == 16) {
      for (int first = 32 * NV; first < sr.span.vecs; first += 32 * NV) {
        sr.load(lane, first);
        sr.template fold_part<ENT>(ps, lane);
        none = none || ps.s == 0.f;
      }
    }
    const SoftmaxPartial q = sr.template finish<ENT>(ps, none, lane);
    if (lane == 0) {
      const float lnS = logf(q.s);
      const float lse = q.m + lnS;
      if (!a_ok) flag_status(p.status, RL_DEV_BAD_TOKEN);
      p.logp_out[r] = a_ok ? za - lse : __int_as_float(0x7fc00000);
      if (p.entropy_out) p.entropy_out[r] = lnS - q.u / q.s;
      if (p.lse_out) p.lse_out[r] = lse;
    }
  }
}

// ------------------------------------------------------------------ forward-only stream
//
// rl_token_logprobs reads each row exactly once and keeps nothing on chip, so it
// needs no cluster: one CTA owns a row at a time (persistent over rows). A
// producer warp streams the CTA's rows as back-to-back chunks through a ring of
// shared-memory stages (bulk copies, full / empty mbarriers); consumer warps fold
// each chunk into per-thread online-softmax partials and, at the end of a row,
// merge them (one named barrier among the consumers per row).
// Stages and chunk size per form, chosen by a sweep on the benchmark batch (bf16, V = 151,936):
// without the entropy 3 x 16 KB (3 CTAs per SM, bound by registers) ran in 6.54 ms per batch
// against 6.80 with 6 x 16 KB (2 CTAs per SM, bound by shared memory); with the entropy
// 4 x 12 KB ran in 7.19 against 7.27 ms (3 x 16 KB: 7.55).
template <bool ENT>
struct FwdCfg {
  static constexpr int kStages = ENT ? 4 : 3;
  static constexpr int kChunkKB = ENT ? 12 : 16;
};

struct ChunkInfo {
  int64_t r;      // row, -1 = end of stream
  int32_t nv;     // whole blocks in the chunk
  int32_t edges;  // elements of the row's partial blocks here: head | tail << 4 | head's place << 8
  int32_t a_at;   // the sampled token's place in the stage, -1: not in this chunk
  int32_t last;   // the row's last chunk: 1, or 2 if the sampled token is out of range
};

// MINB: CTAs per SM the register budget is sized for (2 leaves 64 to 72 registers, 3 CTAs).
template <typename T, int NW, bool ENT, int MINB>
__global__ void __launch_bounds__((NW + 1) * 32, MINB) stream_logprobs_kernel(const StreamArgs p) {
  constexpr int EPV = Vec<T>::N;
  constexpr int NS = FwdCfg<ENT>::kStages;
  constexpr int NC = NW * 32;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full_bar[NS], empty_bar[NS];
  __shared__ ChunkInfo info[NS];
  __shared__ SoftmaxPartial red[2][NW];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t rows = p.rows, V = p.V, ld = p.ld;
  const int CV = p.chunk;
  const T* logits = static_cast<const T*>(p.logits);
  const T* const logits_end = logits + ((rows - 1) * ld + V);
  T* const buf_base = reinterpret_cast<T*>(smem_raw);
  const int edge0 = CV * EPV;  // a stage: the chunk's blocks, the head's block, the tail's block

  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      mbar_init(&full_bar[k], 1);
      mbar_init(&empty_bar[k], NW);
    }
    fence_mbar_init();
  }
  __syncthreads();

  if (warp == NW) {
    // =============================================================== producer warp
    // The sampled ids are fetched 32 rows at a time, one per lane, a batch ahead: the consumers
    // take z_a from the chunk that holds it instead of by two dependent trips at the row's end.
    uint32_t q = 0;
    bool failed = false;
    const int64_t step = gridDim.x;
    auto load_ids = [&](int64_t b0) {
      const int64_t my = b0 + static_cast<int64_t>(lane) * step;
      return my < rows ? p.token_ids[my] : 0;
    };
    int32_t ids = load_ids(blockIdx.x), next_ids = 0;
    int jr = 0;
    for (int64_t r = blockIdx.x; r < rows && !failed; r += step) {
      if (jr == 0) next_ids = load_ids(r + 32 * step);
      const int32_t a = __shfl_sync(0xffffffffu, ids, jr);
      if (++jr == 32) {
        jr = 0;
        ids = next_ids;
      }
      const RowSpan<T> span = row_span<T>(r, ld, V);
      const T* row = logits + r * ld;
      const T* tail = row + (V - span.tail);
      const int nchunk = max(1, (span.vecs + CV - 1) / CV);
      for (int k = 0; k < nchunk; ++k, ++q) {
        const int st = q % NS;
        const uint32_t use = q / NS;
        if (use > 0 && !mbar_wait_bounded(&empty_bar[st], (use - 1) & 1)) {
          failed = true;
          if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
          break;
        }
        const int nv = min(CV, span.vecs - k * CV);
        const bool has_head = k == 0 && span.head > 0, has_tail = k == nchunk - 1 && span.tail > 0;
        const bool head_bulk = has_head && block_inside(row, logits_end);
        const bool tail_bulk = has_tail && block_inside(tail, logits_end);
        T* buf = buf_base + st * p.buf_elems;
        if (has_head && !head_bulk && lane < span.head) buf[edge0 + block_offset(row) + lane] = row[lane];
        if (has_tail && !tail_bulk && lane < span.tail) buf[edge0 + EPV + lane] = tail[lane];
        __syncwarp();
        if (lane == 0) {
          const int hoff = block_offset(row);
          const int rel = a - span.head - k * CV * EPV, tail0 = static_cast<int>(V) - span.tail;
          int a_at = -1;
          if (a >= 0 && a < span.head) {
            if (k == 0) a_at = edge0 + hoff + a;
          } else if (a >= tail0) {
            if (k == nchunk - 1 && a < V) a_at = edge0 + EPV + (a - tail0);
          } else if (rel >= 0 && rel < nv * EPV) {
            a_at = rel;
          }
          info[st] = ChunkInfo{r, nv, (has_head ? span.head : 0) | (has_tail ? span.tail << 4 : 0) | hoff << 8, a_at,
                               k == nchunk - 1 ? (a >= 0 && a < V ? 1 : 2) : 0};
          const uint32_t bytes = static_cast<uint32_t>(nv) * 16u + (head_bulk ? 16u : 0u) + (tail_bulk ? 16u : 0u);
          if (bytes > 0) {
            mbar_arrive_expect_tx(&full_bar[st], bytes);
            if (nv > 0) bulk_g2s(buf, row + span.head + static_cast<int64_t>(k) * CV * EPV, nv * 16u, &full_bar[st]);
            if (head_bulk) bulk_g2s(buf + edge0, row - block_offset(row), 16u, &full_bar[st]);
            if (tail_bulk) bulk_g2s(buf + edge0 + EPV, tail, 16u, &full_bar[st]);
          } else {
            mbar_arrive(&full_bar[st]);
          }
        }
      }
    }
    if (!failed) {
      const int st = q % NS;
      const uint32_t use = q / NS;
      if (use > 0 && !mbar_wait_bounded(&empty_bar[st], (use - 1) & 1)) {
        if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
      } else if (lane == 0) {
        info[st].r = -1;
        mbar_arrive(&full_bar[st]);
      }
    }
  } else {
    // =============================================================== consumer warps
    SoftmaxPartial ps{RL_NEG_INF, 0.f, 0.f};
    float za = 0.f;  // the row's z_a (thread 0)
    uint32_t row_it = 0;
    for (uint32_t q = 0;; ++q) {
      const int st = q % NS;
      if (!mbar_wait_bounded(&full_bar[st], (q / NS) & 1)) {
        if (tid == 0) flag_status(p.status, RL_DEV_TIMEOUT);
        break;
      }
      const ChunkInfo ci = info[st];
      if (ci.r < 0) break;
      const T* buf = buf_base + st * p.buf_elems;
      const int nv = ci.nv;
      {
        // only as many vectors per thread as the chunk has: a row's last chunk is often short
        constexpr int KV = (FwdCfg<ENT>::kChunkKB * 1024 / 16 + NC - 1) / NC;  // vectors per thread per chunk
        static_assert(KV <= 4, "the cases below");
        const uint32_t pad = Vec<T>::kPadWord;
        auto reload = [&](int k) {
          const int j = tid + k * NC;
          return j < nv ? reinterpret_cast<const uint4*>(buf)[j] : make_uint4(pad, pad, pad, pad);
        };
        auto fold_n = [&](auto n) {
          uint4 x[decltype(n)::value];
#pragma unroll
          for (int k = 0; k < decltype(n)::value; ++k) x[k] = reload(k);
          fold_block<T, ENT>(ps, x, reload);
        };
        if (KV > 3 && nv > 3 * NC) fold_n(std::integral_constant<int, 4>{});
        else if (KV > 2 && nv > 2 * NC) fold_n(std::integral_constant<int, 3>{});
        else if (nv > NC) fold_n(std::integral_constant<int, 2>{});
        else if (nv > 0) fold_n(std::integral_constant<int, 1>{});
      }
      // the row's partial blocks: the head's elements by the first warp, the tail's by the second
      if (warp < 2 && (ci.edges & 0xFF) != 0) {
        const int at = edge0 + (warp == 0 ? (ci.edges >> 8) + lane : EPV + lane);
        if (lane < (warp == 0 ? ci.edges & 15 : (ci.edges >> 4) & 15)) {
          const float z = Vec<T>::to_f(buf[at]);
          if (z != RL_NEG_INF) {
            raise_max<ENT>(ps, z);
            accumulate<ENT>(ps, z, -ps.m * kLog2e);
          }
        }
      }
      if (tid == 0 && ci.a_at >= 0) za = Vec<T>::to_f(buf[ci.a_at]);
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty_bar[st]);
      if (ci.last) {
        // ---- end of row ci.r: merge the consumers' partials
        const int par = row_it & 1;
        ps = warp_merge<ENT>(ps);
        if (lane == 0) red[par][warp] = ps;
        asm volatile("bar.sync 1, %0;" :: "n"(NC) : "memory");
        if (warp == 0) {
          SoftmaxPartial qq = lane < NW ? red[par][lane] : SoftmaxPartial{RL_NEG_INF, 0.f, 0.f};
          qq = warp_merge<ENT>(qq);
          if (lane == 0) {
            const int64_t r = ci.r;
            const float lnS = logf(qq.s);
            const float lse = qq.m + lnS;
            const bool a_ok = ci.last == 1;
            if (!a_ok) flag_status(p.status, RL_DEV_BAD_TOKEN);
            p.logp_out[r] = a_ok ? za - lse : __int_as_float(0x7fc00000);
            if (p.entropy_out) p.entropy_out[r] = lnS - qq.u / qq.s;
            if (p.lse_out) p.lse_out[r] = lse;
          }
        }
        ps = SoftmaxPartial{RL_NEG_INF, 0.f, 0.f};
        ++row_it;
      }
    }
  }
}

// ------------------------------------------------------------------ host side

constexpr int64_t kMaxSliceBytes = 100 * 1024;

struct Plan {
  int C;
  int64_t slice, buf_elems;
  size_t smem;
};

// A row of V elements of es bytes cut into C slices.
static Plan cut(int64_t V, int es, int C) {
  const int64_t epv = 16 / es;
  const int64_t slice = ((V + C - 1) / C + epv - 1) / epv * epv;
  const int64_t stride_bytes = (slice * es + 32 + 127) / 128 * 128;  // and the row's two partial blocks
  return Plan{C, slice, stride_bytes / es, static_cast<size_t>(RL_STAGES * stride_bytes)};
}

// Smallest cluster whose slices are at most target_bytes (or, at 16 CTAs, at most 100 KB).
static bool make_plan(int64_t V, int es, Plan* out, int64_t target_bytes = 40 * 1024) {
  for (int C = 1; C <= 16; ++C) {
    *out = cut(V, es, C);
    const int64_t bytes = out->slice * es;
    if (bytes <= target_bytes || (C == 16 && bytes <= kMaxSliceBytes)) return true;
  }
  return false;
}

// Configure a kernel once per (kernel, device): dynamic shared memory up to the
// largest request so far, and non-portable cluster sizes allowed.
static rl_status configure(const void* kern, int dev, size_t smem) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, size_t> smem_attr;
  std::lock_guard<std::mutex> lock(mu);
  auto ka = std::make_pair(kern, dev);
  auto ita = smem_attr.find(ka);
  if (ita == smem_attr.end() || ita->second < smem) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(max dynamic smem)");
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(non-portable cluster)");
    smem_attr[ka] = smem;
  }
  return RL_OK;
}

static rl_status launch_clusters(void (*kern)(RowArgs), int threads, const RowArgs& args, const Plan& plan,
                                 cudaStream_t s, int64_t* n_clusters_out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  rl_status st = configure(reinterpret_cast<const void*>(kern), dev, plan.smem);
  if (st != RL_OK) return st;

  static std::mutex mu;
  static std::map<std::tuple<const void*, int, int, size_t>, int> cache;
  int max_clusters = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto key = std::make_tuple(reinterpret_cast<const void*>(kern), dev, plan.C, plan.smem);
    auto itc = cache.find(key);
    if (itc != cache.end()) {
      max_clusters = itc->second;
    } else {
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = plan.C;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(plan.C * 1024, 1, 1);
      cfg.blockDim = dim3(threads, 1, 1);
      cfg.dynamicSmemBytes = plan.smem;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      e = cudaOccupancyMaxActiveClusters(&max_clusters, kern, &cfg);
      if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveClusters");
      if (max_clusters <= 0) return set_error(RL_ERR_UNSUPPORTED, "no cluster of this shape fits on the device");
      cache[key] = max_clusters;
    }
  }
  const int64_t n_clusters = std::max<int64_t>(1, std::min<int64_t>(max_clusters, args.rows));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = plan.C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(n_clusters * plan.C), 1, 1);
  cfg.blockDim = dim3(threads, 1, 1);
  cfg.dynamicSmemBytes = plan.smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, kern, args);
  if (e != cudaSuccess) return cuda_error(e, "cudaLaunchKernelEx(rows_kernel)");
  if (n_clusters_out) *n_clusters_out = n_clusters;
  return RL_OK;
}

template <typename T, int NW, bool ENT, int HOLDV, int MINB, bool SHIFT = false>
static rl_status launch_rows(const RowArgs& args, const Plan& plan, cudaStream_t s, int64_t* n_clusters_out) {
  return launch_clusters(rows_kernel<T, NW, ENT, HOLDV, MINB, SHIFT>, (NW + 1) * 32, args, plan, s, n_clusters_out);
}

template <bool ENT>
static rl_status launch_f32(const RowArgs& args, const Plan& plan, cudaStream_t s, int64_t* n_clusters_out) {
  return launch_clusters(rows_f32_kernel<ENT>, (kF32Warps + 1) * 32, args, plan, s, n_clusters_out);
}

// Shapes of rows_kernel: consumer warps, 16-byte vectors each of their threads holds, CTAs per SM.
struct Shape {
  int warps, hold, per_sm;
};
constexpr Shape kShapes[] = {{8, 10, 2}, {8, 6, 3}, {4, 10, 4}, {4, 5, 5}, {16, 10, 1}, {19, 11, 1}};

// The shape and the cluster width for rows of up to V entries (above the entry before). The time a CTA
// takes per row, 2.5 to 4 us, is a chain of waits (the slice, the exchange, the merges) that depends
// little on how full its slice is, so what counts is how many bytes of rows are resident, up to 10 to 15
// MB, past which reads and writes of more rows at once slow the memory down: which of the shapes comes
// closest changes with every slice that a cluster more or less brings, by no simple law. So the lines are
// where the measurements cross, or where a row outgrows its slices. Measured: every shape at its three
// narrowest widths, 146 vocabularies of 4,104 to 819,200 bf16 entries and 39 of 129,032 to 409,600 fp32
// ones (0.8 GB of logits), all rows trained without and with the entropy, and 62% of them trained in
// spans; a crossing that one of the three loses by more than 2% is left out. In the mean of the three
// the choice is 0.8% from the fastest on average and 7% at most (fp32: 0.1% and 2%). GB/s read and
// written, all rows trained without the entropy, against one shape for all (8 x 10 at 2 CTAs per SM,
// slices of 20 to 40 KB): V = 4,160 4,810 (1,682), 8,192 5,560 (3,156), 25,600 5,880 (4,614), 32,000 6,190
// (5,503), 65,536 6,110 (5,301), 128,256 6,180 (5,077), 151,936 6,220 (5,625), 262,144 5,490 (4,729). The
// number of rows does not enter: a row's results do not depend on the size of its microbatch (bf16 rows
// with a leading dimension that is no multiple of 8 are cut where memory blocks end, so the order of
// their sums depends on r ld mod 8).
struct Pick {
  int32_t V;
  int8_t shape, C;
};
constexpr Pick kPicksBf16[] = {
    {5120, 3, 1}, {8816, 2, 1}, {12288, 1, 1}, {19320, 0, 1}, {22800, 1, 2}, {26800, 2, 3}, {29720, 0, 2},
    {36552, 4, 1}, {41440, 5, 1}, {44440, 2, 5}, {47624, 1, 4}, {59768, 2, 6}, {68608, 0, 4},
    {78848, 4, 2}, {82888, 5, 2}, {102400, 2, 10}, {108536, 2, 11}, {122880, 0, 6}, {133120, 2, 13},
    {143360, 0, 7}, {163840, 4, 4}, {184320, 0, 9}, {204800, 5, 4}, {256000, 5, 5}, {307200, 5, 6},
    {368640, 4, 9}, {409600, 4, 10}, {460800, 5, 9}, {512000, 5, 10}, {655360, 4, 16}, {768000, 5, 15},
    {819200, 5, 16},
};
constexpr Pick kPicksF32[] = {
    {153600, 5, 6}, {184320, 4, 9}, {197488, 4, 10}, {204800, 5, 8}, {230400, 5, 9}, {256000, 5, 10},
    {286720, 4, 14}, {327680, 4, 16}, {343992, 5, 14}, {384000, 5, 15}, {409600, 5, 16},
};

// A CTA's slice of a row fits the registers that its shape holds it in, and a stage.
constexpr bool fits(const Pick& p, int es) {
  const int64_t epv = 16 / es, bytes = ((p.V + p.C - 1) / p.C + epv - 1) / epv * 16;
  return bytes <= static_cast<int64_t>(kShapes[p.shape].warps) * 32 * kShapes[p.shape].hold * 16 &&
         bytes <= kMaxSliceBytes;
}
template <int N>
constexpr bool all_fit(const Pick (&t)[N], int es) {
  for (int k = 0; k < N; ++k)
    if (!fits(t[k], es) || (k > 0 && t[k].V <= t[k - 1].V)) return false;
  return static_cast<int64_t>(t[N - 1].V) * es == 16 * kMaxSliceBytes;
}
static_assert(all_fit(kPicksBf16, 2) && all_fit(kPicksF32, 4), "every row up to the largest has a shape that holds it");

template <int N>
static int pick_shape(const Pick (&t)[N], int64_t V, int es, Plan* plan) {
  for (const Pick& p : t)
    if (V <= p.V) {
      *plan = cut(V, es, p.C);
      return p.shape;
    }
  return -1;
}

// Launches a short-row kernel: as many CTAs as fit on the GPU at once, at most one warp per row.
template <typename Args>
static rl_status launch_small(void (*kern)(Args), const Args& args, cudaStream_t s) {
  constexpr int kThreads = kSmallWarps * 32;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, int64_t> grid_cache;
  int64_t grid = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto key = std::make_pair(reinterpret_cast<const void*>(kern), dev);
    auto it = grid_cache.find(key);
    if (it != grid_cache.end()) {
      grid = it->second;
    } else {
      int per_sm = 0, sms = 0;
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, 0);
      if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
      e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      if (e != cudaSuccess) return cuda_error(e, "cudaDeviceGetAttribute");
      if (per_sm <= 0) return set_error(RL_ERR_UNSUPPORTED, "the short-row kernel does not fit on an SM");
      grid = static_cast<int64_t>(per_sm) * sms;
      grid_cache[key] = grid;
    }
  }
  const int64_t blocks = std::min<int64_t>(grid, (args.rows + kSmallWarps - 1) / kSmallWarps);
  kern<<<static_cast<unsigned>(blocks), kThreads, 0, s>>>(args);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, "short-row kernel launch");
  return RL_OK;
}

// Blocks a lane holds of a short row (a row of n bytes has at most n / 16 whole blocks).
static int small_blocks(int64_t row_bytes) { return row_bytes <= 2048 ? 4 : row_bytes <= 4096 ? 8 : 16; }

template <typename T>
static rl_status dispatch_loss(bool ent, RowArgs args, int64_t V, cudaStream_t s, int64_t* n_clusters) {
  // rows of at most 8 KB: a warp per row
  const int64_t row_bytes = V * static_cast<int64_t>(sizeof(T));
  if (row_bytes <= kSmallRowBytes) {
    *n_clusters = 0;
    switch (small_blocks(row_bytes)) {
      case 4: return launch_small(ent ? small_rows_kernel<T, true, 4> : small_rows_kernel<T, false, 4>, args, s);
      case 8: return launch_small(ent ? small_rows_kernel<T, true, 8> : small_rows_kernel<T, false, 8>, args, s);
      default: return launch_small(ent ? small_rows_kernel<T, true, 16> : small_rows_kernel<T, false, 16>, args, s);
    }
  }
  auto run = [&](const Plan& plan, auto launcher) {
    args.slice = plan.slice;
    args.buf_elems = plan.buf_elems;
    return launcher(args, plan, s, n_clusters);
  };
  Plan plan = {};
  if constexpr (sizeof(T) == 4) {
    // fp32: slices of at most 30 KB on 3 CTAs per SM (another cut would change the order of the sums
    // and with it the last bits), wider rows by kPicksF32
    const bool shift = args.ld % 4 != 0;
    if (make_plan(V, 4, &plan, 30 * 1024) && plan.slice * 4 <= kF32Hold * kF32Warps * 32 * 16) {
      if (!shift) return ent ? run(plan, launch_f32<true>) : run(plan, launch_f32<false>);
      return ent ? run(plan, launch_rows<T, 7, true, 9, 3, true>) : run(plan, launch_rows<T, 7, false, 9, 3, true>);
    }
#define RL_RUN(K, SHIFT) \
  (ent ? run(plan, launch_rows<T, kShapes[K].warps, true, kShapes[K].hold, kShapes[K].per_sm, SHIFT>) \
       : run(plan, launch_rows<T, kShapes[K].warps, false, kShapes[K].hold, kShapes[K].per_sm, SHIFT>))
    switch (pick_shape(kPicksF32, V, 4, &plan)) {
      case 4: return shift ? RL_RUN(4, true) : RL_RUN(4, false);
      case 5: return shift ? RL_RUN(5, true) : RL_RUN(5, false);
    }
  } else {
    switch (pick_shape(kPicksBf16, V, 2, &plan)) {
      case 0: return RL_RUN(0, false);
      case 1: return RL_RUN(1, false);
      case 2: return RL_RUN(2, false);
      case 3: return RL_RUN(3, false);
      case 4: return RL_RUN(4, false);
      case 5: return RL_RUN(5, false);
    }
#undef RL_RUN
  }
  return set_error(RL_ERR_UNSUPPORTED, "rl_policy_loss_fwd_bwd: row too large");
}

constexpr int kFwdWarps = 8;

// CTAs of a streaming kernel that fit on the GPU at once.
static rl_status stream_grid(void (*kern)(StreamArgs), size_t smem, int* grid) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  rl_status st = configure(reinterpret_cast<const void*>(kern), dev, smem);
  if (st != RL_OK) return st;
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, int> cache;
  std::lock_guard<std::mutex> lock(mu);
  auto key = std::make_pair(reinterpret_cast<const void*>(kern), dev);
  auto it = cache.find(key);
  if (it == cache.end()) {
    int per_sm = 0, sms = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, (kFwdWarps + 1) * 32, smem);
    if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_error(e, "cudaDeviceGetAttribute");
    if (per_sm <= 0) return set_error(RL_ERR_UNSUPPORTED, "stream kernel does not fit on an SM");
    it = cache.emplace(key, per_sm * sms).first;
  }
  *grid = it->second;
  return RL_OK;
}

template <typename T, bool ENT>
static rl_status launch_stream(StreamArgs args, cudaStream_t s) {
  const int64_t row_bytes = args.V * static_cast<int64_t>(sizeof(T));
  if (row_bytes <= (sizeof(T) == 2 && ENT ? 4 : 2) * kSmallRowBytes) {
    switch (small_blocks(row_bytes)) {
      case 4: return launch_small(small_logprobs_kernel<T, ENT, 4>, args, s);
      case 8: return launch_small(small_logprobs_kernel<T, ENT, 8>, args, s);
      default: return launch_small(small_logprobs_kernel<T, ENT, 16>, args, s);
    }
  }
  args.chunk = FwdCfg<ENT>::kChunkKB * 1024 / 16;
  // the chunk, then the row's two partial blocks, to a multiple of 128 bytes
  args.buf_elems = (static_cast<int64_t>(args.chunk) * 16 + 128) / static_cast<int64_t>(sizeof(T));
  const size_t smem = static_cast<size_t>(FwdCfg<ENT>::kStages) * args.buf_elems * sizeof(T);
  auto kern = stream_logprobs_kernel<T, kFwdWarps, ENT, 2>;
  int grid = 0;
  rl_status st = stream_grid(kern, smem, &grid);
  if (st != RL_OK) return st;
  if constexpr (sizeof(T) == 4) {
    // fp32 rows are long, and few of them may fill their last round of the grid badly: with 4 CTAs per SM
    // where that takes fewer places. 0.8 GB of rows: 1,316 rows of 151,936 entries 116 us on 3 CTAs per SM
    // (1,368 places) and 125 on 4 (1,824), 999 of 200,064 126 and 118, 500 of 400,000 147 and 117.
    auto kern4 = stream_logprobs_kernel<T, kFwdWarps, ENT, 4>;
    int grid4 = 0;
    st = stream_grid(kern4, smem, &grid4);
    if (st != RL_OK) return st;
    auto places = [&](int64_t g) { return (args.rows + g - 1) / g * g; };
    if (places(grid4) < places(grid)) {
      kern = kern4;
      grid = grid4;
    }
  }
  const unsigned blocks = static_cast<unsigned>(std::min<int64_t>(grid, args.rows));
  kern<<<blocks, (kFwdWarps + 1) * 32, smem, s>>>(args);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, "stream_logprobs_kernel launch");
  return RL_OK;
}

static rl_status check_rows_args(const char* fn, const void* logits, rl_dtype dt, int64_t rows, int64_t V,
                                 int64_t ld, const void* ws, size_t ws_bytes, Plan* plan, int* es) {
  if (dt != RL_BF16 && dt != RL_F32) return set_error(RL_ERR_INVALID_ARG, std::string(fn) + ": unknown dtype");
  if (rows < 0 || V < 1 || ld < V)
    return set_error(RL_ERR_INVALID_ARG, std::string(fn) + ": need rows >= 0, V >= 1, ld >= V");
  if (!ws) return set_error(RL_ERR_INVALID_ARG, std::string(fn) + ": ws is NULL");
  if (ws_bytes < rl_workspace_size(rows, V, 0))
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL, std::string(fn) + ": workspace smaller than rl_workspace_size(rows, V, 0)");
  if (!aligned16(ws)) return set_error(RL_ERR_ALIGNMENT, std::string(fn) + ": ws not 16-byte aligned");
  if (rows > 0 && !logits) return set_error(RL_ERR_INVALID_ARG, std::string(fn) + ": logits is NULL");
  if (logits && !aligned16(logits)) return set_error(RL_ERR_ALIGNMENT, std::string(fn) + ": logits not 16-byte aligned");
  if (V > INT32_MAX) return set_error(RL_ERR_UNSUPPORTED, std::string(fn) + ": V above 2^31 - 1");
  *es = dt == RL_BF16 ? 2 : 4;
  if (!make_plan(V, *es, plan))
    return set_error(RL_ERR_UNSUPPORTED, std::string(fn) + ": vocabulary row larger than 16 x 100 KB");
  return RL_OK;
}

}  // namespace rl

extern "C" rl_status rl_token_logprobs(const void* logits, rl_dtype dtype, int64_t rows, int64_t V, int64_t ld,
                                       const int32_t* token_ids, float* logp_out, float* entropy_out,
                                       float* lse_out, void* ws, size_t ws_bytes, rl_stream_t stream) {
  using namespace rl;
  clear_error();
  Plan plan;
  int es = 0;
  rl_status st = check_rows_args("rl_token_logprobs", logits, dtype, rows, V, ld, ws, ws_bytes, &plan, &es);
  if (st != RL_OK) return st;
  if (rows == 0) return RL_OK;
  if (!token_ids || !logp_out) return set_error(RL_ERR_INVALID_ARG, "rl_token_logprobs: NULL array argument");
  StreamArgs a = {};
  a.logits = logits;
  a.rows = rows;
  a.V = V;
  a.ld = ld;
  a.token_ids = token_ids;
  a.logp_out = logp_out;
  a.entropy_out = entropy_out;
  a.lse_out = lse_out;
  a.status = reinterpret_cast<int32_t*>(ws);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (dtype == RL_BF16)
    return entropy_out ? launch_stream<uint16_t, true>(a, s) : launch_stream<uint16_t, false>(a, s);
  return entropy_out ? launch_stream<float, true>(a, s) : launch_stream<float, false>(a, s);
}

extern "C" rl_status rl_policy_loss_fwd_bwd(const void* logits, rl_dtype dtype, int64_t rows, int64_t V,
                                            int64_t ld, const int32_t* token_ids, const uint8_t* mask,
                                            const int32_t* token_traj, int32_t n_traj, const float* adv,
                                            const float* coef, const float* old_logp, const float* ref_logp,
                                            const float* rollout_logp, const rl_loss_params* params,
                                            void* grad_out, double* loss_accum, float* token_stats, void* ws,
                                            size_t ws_bytes, rl_stream_t stream) {
  using namespace rl;
  clear_error();
  Plan plan;
  int es = 0;
  rl_status st = check_rows_args("rl_policy_loss_fwd_bwd", logits, dtype, rows, V, ld, ws, ws_bytes, &plan, &es);
  if (st != RL_OK) return st;
  if (!params) return set_error(RL_ERR_INVALID_ARG, "rl_policy_loss_fwd_bwd: params is NULL");
  if (!(params->clip_eps_low >= 0.f) || !(params->clip_eps_high >= 0.f))
    return set_error(RL_ERR_INVALID_ARG, "rl_policy_loss_fwd_bwd: clip eps must be >= 0");
  if (params->kl_estimator != 0 && params->kl_estimator != 3)
    return set_error(RL_ERR_UNSUPPORTED, "rl_policy_loss_fwd_bwd: kl_estimator must be 0 or 3");
  if (!loss_accum) return set_error(RL_ERR_INVALID_ARG, "rl_policy_loss_fwd_bwd: loss_accum is NULL");
  if (n_traj < 0) return set_error(RL_ERR_INVALID_ARG, "rl_policy_loss_fwd_bwd: n_traj < 0");
  if (rows == 0) return RL_OK;
  if (!token_ids || !mask || !token_traj || !old_logp || !grad_out || (n_traj > 0 && (!adv || !coef)) ||
      (params->token_level_adv && !adv))
    return set_error(RL_ERR_INVALID_ARG, "rl_policy_loss_fwd_bwd: NULL array argument");
  if (params->token_level_adv != 0 && params->token_level_adv != 1)
    return set_error(RL_ERR_INVALID_ARG, "rl_policy_loss_fwd_bwd: token_level_adv must be 0 or 1");
  if (!aligned16(grad_out)) return set_error(RL_ERR_ALIGNMENT, "rl_policy_loss_fwd_bwd: grad_out not 16-byte aligned");
  const bool kl_on = params->kl_estimator == 3 && params->kl_coef != 0.f && ref_logp != nullptr;
  RowArgs a = {};
  a.logits = logits;
  a.grad = grad_out;
  a.rows = rows;
  a.V = V;
  a.ld = ld;
  a.token_ids = token_ids;
  a.mask = mask;
  a.token_traj = token_traj;
  a.n_traj = n_traj;
  a.adv = adv;
  a.coef = coef;
  a.old_logp = old_logp;
  a.ref_logp = kl_on ? ref_logp : nullptr;
  a.rollout_logp = rollout_logp;
  a.clip_lo = 1.f - params->clip_eps_low;
  a.clip_hi = 1.f + params->clip_eps_high;
  a.beta = kl_on ? params->kl_coef : 0.f;
  a.alpha = params->entropy_coef;
  a.tis_cap = rollout_logp ? params->tis_cap : 0.f;
  a.adv_per_row = params->token_level_adv;
  double* row_loss = reinterpret_cast<double*>(static_cast<char*>(ws) + ws_row_loss_offset());
  a.row_loss = row_loss;
  a.loss_accum = loss_accum;
  a.done = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + kWsDoneOffset);
  a.token_stats = token_stats;
  a.status = reinterpret_cast<int32_t*>(ws);
  const bool ent = params->entropy_coef != 0.f || token_stats != nullptr;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int64_t n_clusters = 0;
  st = dtype == RL_BF16 ? dispatch_loss<uint16_t>(ent, a, V, s, &n_clusters)
                        : dispatch_loss<float>(ent, a, V, s, &n_clusters);
  return st;  // the kernel's last cluster has added the loss into loss_accum
}
