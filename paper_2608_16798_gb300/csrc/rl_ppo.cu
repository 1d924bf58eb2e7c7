// PPO parts of the method (Sec. 2.3.1, Sec. 2.3.4): the masked generalised advantage
// estimate over packed ragged trajectories and the masked value loss.
//
//   gae_kernel         a warp per trajectory of up to kWarpTokens tokens, a CTA per longer one.
//                      The estimate is the backward
//                      affine recurrence x_t = a_t x_{t+1} + b_t inside the trajectory
//                      (x past its end = 0), evaluated chunk by chunk from the end: each
//                      thread composes its 4 tokens' maps, a warp- or block-wide suffix scan of
//                      the composed maps gives every thread its entry value, and the chunk's
//                      first value carries into the next chunk down.
//                        printed reading  a_t = gamma lambda,
//                                         b_t = M_t (r_t + gamma M_{t+1} V_{t+1} - V_t)
//                        skip reading     a_t = M_t ? gamma lambda : 1,
//                                         b_t = M_t (r_t + gamma Vn_{t+1} - V_t), with
//                                         Vn_{t+1} the value of the next trainable token,
//                                         itself the suffix scan of the selection map
//                                         x_t = M_t ? V_t : x_{t+1} (exact in fp32)
//                      R_i is added at the token with M_t = 1 that has no later one: the scan of
//                      "is there a trainable token above" rides along.
//   value_loss_kernel  per token: c M (V - G)^2, added per CTA in a fixed order into one
//                      partial per CTA, and dV = 2 c M (V - G); the last CTA to finish adds
//                      the partials, in a fixed order, into the caller's accumulator.
//   rollout_adv_kernel A_t = R_i - V_t, G_t = R_i per token for tokens in any order (the
//                      gamma = lambda = 1 form of Sec. 2.3.4, which also holds on the shared
//                      prefixes of a rollout's prefix tree).
//
// Both touch a few bytes per token (mask, values, rewards, outputs) and are latency- or
// launch-bound next to the logits stream.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "rl_device.cuh"
#include "rl_host.h"

namespace rl {
namespace ppo {

constexpr int kThreads = 256;
constexpr int kPer = 4;                  // consecutive tokens per thread
constexpr int kWarps = kThreads / 32;

// x -> a x + b
struct Affine {
  float a, b;
};

// outer(inner(x)): inner is applied first (it covers the later positions).
__device__ __forceinline__ Affine compose(Affine outer, Affine inner) {
  return Affine{outer.a * inner.a, fmaf(outer.a, inner.b, outer.b)};
}

constexpr int kWarpTokens = 512;  // longest trajectory one warp takes

struct GaeArgs {
  int32_t n_traj;
  int32_t per_cta;  // trajectories of a CTA (at most kWarps)
  const int64_t* offs;
  int64_t T;
  const uint8_t* mask;
  const float* values;
  const float* token_rewards;  // [T] or null
  const float* traj_rewards;   // [n_traj] or null: R_i at the last trainable token
  float gamma, lam;
  int32_t skip;
  float* adv;
  float* ret;  // or null
  int32_t* status;
};

// The same scan for one warp (W = 1) or the whole CTA (W = kWarps). Every thread passes the
// composition of its own tokens' maps (`mine`, mapping the value just above its tokens to the
// value at its first token) and the value above the whole chunk (`top`, the same in every thread);
// returns the value just above this thread's tokens, and in `low` (the same in every thread) the
// value at the chunk's first token. `sh` holds kWarps maps; the caller alternates between two of
// them, so one barrier per scan suffices.
template <int W>
__device__ __forceinline__ float suffix_entry(Affine mine, float top, Affine* sh, float& low) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // inclusive suffix within the warp: S_k = F_k o F_{k+1} o ... o F_31
  Affine s = mine;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const float oa = __shfl_down_sync(0xffffffffu, s.a, off);
    const float ob = __shfl_down_sync(0xffffffffu, s.b, off);
    if (lane + off < 32) s = compose(s, Affine{oa, ob});
  }
  // value above this warp: the later warps' totals applied to `top`, highest first
  float above_warp = top;
  if (W > 1) {
    if (lane == 0) sh[warp] = s;
    __syncthreads();
    low = top;
#pragma unroll
    for (int w = W - 1; w >= 0; --w) {
      if (w == warp) above_warp = low;
      low = fmaf(sh[w].a, low, sh[w].b);
    }
  } else {
    low = fmaf(__shfl_sync(0xffffffffu, s.a, 0), top, __shfl_sync(0xffffffffu, s.b, 0));
  }
  // exclusive suffix within the warp: S_{k+1} applied to the warp's entry value
  const float na = __shfl_down_sync(0xffffffffu, s.a, 1);
  const float nb = __shfl_down_sync(0xffffffffu, s.b, 1);
  return lane == 31 ? above_warp : fmaf(na, above_warp, nb);
}

// One chunk's inputs of a thread (kPer consecutive tokens from t0), loaded a chunk ahead.
struct GaeTokens {
  bool M[kPer];
  float V[kPer], r[kPer];
};

__device__ __forceinline__ GaeTokens load_tokens(const GaeArgs& p, int64_t t0, int64_t c1) {
  GaeTokens x;
  uint8_t m[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int64_t t = t0 + j;
    const bool in = t < c1;
    m[j] = in ? p.mask[t] : 0;
    x.V[j] = in ? p.values[t] : 0.f;
    x.r[j] = (in && p.token_rewards) ? p.token_rewards[t] : 0.f;
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j) x.M[j] = m[j] != 0;
  return x;
}

// Trajectory [s, e) by one warp (W = 1) or the whole CTA (W = kWarps). Two barriers per chunk of
// the CTA form (one per scan).
template <int W>
__device__ __forceinline__ void gae_trajectory(const GaeArgs& p, int32_t i, int64_t s, int64_t e, Affine (*sh)[kWarps],
                                               uint32_t* sh_any) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tid = W > 1 ? static_cast<int>(threadIdx.x) : lane;
  constexpr int kStep = W * 32 * kPer;
  const float gl = p.gamma * p.lam;
  const float Ri = p.traj_rewards ? p.traj_rewards[i] : 0.f;
  float carry_x = 0.f;    // recurrence value at the first position above the chunk
  float carry_vn = 0.f;   // value of the first trainable token above it (skip reading) ...
  float edge_vn = 0.f;    // ... or M V of the first token above it (printed reading)
  bool seen = false;      // a trainable token lies above the chunk
  GaeTokens cur = load_tokens(p, (e - kStep > s ? e - kStep : s) + static_cast<int64_t>(tid) * kPer, e), nxt;
  for (int64_t c1 = e; c1 > s; c1 -= kStep) {
    const int64_t c0 = c1 - kStep > s ? c1 - kStep : s;
    const int64_t t0 = c0 + static_cast<int64_t>(tid) * kPer;
    const int64_t n1 = c1 - kStep, n0 = n1 - kStep > s ? n1 - kStep : s;  // the next chunk down
    nxt = cur;
    if (n1 > s) nxt = load_tokens(p, n0 + static_cast<int64_t>(tid) * kPer, n1);
    const GaeTokens& x = cur;
    float a[kPer], b[kPer], r[kPer];
    // ---- where R_i goes: the last trainable token of the trajectory, in the first chunk from
    // the end that has one
    bool any = false;
#pragma unroll
    for (int j = 0; j < kPer; ++j) any |= x.M[j];
    const unsigned in_warp = __ballot_sync(0xffffffffu, any);
    if (W > 1 && lane == 0) sh_any[warp] = in_warp;  // read after the next barrier
    bool above = (in_warp >> lane) > 1u;             // a later lane of this warp has one
#pragma unroll
    for (int j = 0; j < kPer; ++j) r[j] = x.r[j];
    float vn = 0.f, low;
    if (p.skip) {
      // Vn above each token: suffix scan of the selection maps
      Affine f{1.f, 0.f};
#pragma unroll
      for (int j = kPer - 1; j >= 0; --j) f = compose(x.M[j] ? Affine{0.f, x.V[j]} : Affine{1.f, 0.f}, f);
      vn = suffix_entry<W>(f, carry_vn, sh[0], low);
      carry_vn = low;
    } else {
      // M V of the token above this thread's last one: the next lane's or warp's first, or, for the
      // thread that holds the chunk's last token, the first of the chunk above
      const float first = x.M[0] ? x.V[0] : 0.f;
      const float edge = edge_vn;
      vn = __shfl_down_sync(0xffffffffu, first, 1);
      if (W > 1) {
        if (lane == 0) sh[0][warp] = Affine{first, 0.f};
        __syncthreads();
        if (lane == 31 && warp + 1 < W) vn = sh[0][warp + 1].a;
        edge_vn = sh[0][0].a;
      } else {
        edge_vn = __shfl_sync(0xffffffffu, first, 0);
      }
      if (t0 + kPer >= c1) vn = edge;
    }
    bool any_chunk = in_warp != 0u;
    if (W > 1) {
      any_chunk = false;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const bool h = sh_any[w] != 0u;
        any_chunk |= h;
        above |= h && w > warp;
      }
    }
    if (any && !above && !seen) {
      bool put = false;
#pragma unroll
      for (int j = kPer - 1; j >= 0; --j)
        if (x.M[j] && !put) {
          r[j] += Ri;
          put = true;
        }
    }
    seen |= any_chunk;
#pragma unroll
    for (int j = kPer - 1; j >= 0; --j) {
      if (p.skip) {
        a[j] = x.M[j] ? gl : 1.f;
        b[j] = x.M[j] ? (r[j] + fmaf(p.gamma, vn, -x.V[j])) : 0.f;
        if (x.M[j]) vn = x.V[j];
      } else {
        const bool in = t0 + j < c1;  // past the chunk: identity
        a[j] = in ? gl : 1.f;
        b[j] = x.M[j] ? (r[j] + fmaf(p.gamma, vn, -x.V[j])) : 0.f;
        if (in) vn = x.M[j] ? x.V[j] : 0.f;
      }
    }
    Affine f{1.f, 0.f};
#pragma unroll
    for (int j = kPer - 1; j >= 0; --j) f = compose(Affine{a[j], b[j]}, f);
    float y = suffix_entry<W>(f, carry_x, sh[1], low);
    carry_x = low;
#pragma unroll
    for (int j = kPer - 1; j >= 0; --j) {
      y = fmaf(a[j], y, b[j]);
      const int64_t t = t0 + j;
      if (t < c1) {
        p.adv[t] = x.M[j] ? y : 0.f;
        if (p.ret) p.ret[t] = x.M[j] ? y + x.V[j] : 0.f;
      }
    }
    cur = nxt;
  }
}

// Latency-bound: a chunk is a trip to memory (hidden behind the chunk before it) and two scans.
// 16,384 trajectories of 8 tokens: 89 us with a CTA each, 13.7 us; 512 of 512 to 8,192: 23.8, 20.4.
// A CTA takes p.per_cta neighbouring trajectories, each of at most kWarpTokens tokens by a warp of
// its own, which meets no barrier; the longer ones are taken by the whole CTA afterwards.
__global__ void __launch_bounds__(kThreads) gae_kernel(const GaeArgs p) {
  __shared__ Affine sh[2][kWarps];
  __shared__ uint32_t sh_any[kWarps];
  __shared__ int64_t span[kWarps][2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * p.per_cta; base < p.n_traj;
       base += static_cast<int64_t>(gridDim.x) * p.per_cta) {
    const int here = static_cast<int>(min(static_cast<int64_t>(p.per_cta), p.n_traj - base));
    if (warp < here) {
      const int32_t i = static_cast<int32_t>(base) + warp;
      const int64_t s = p.offs[i], e = p.offs[i + 1];
      const bool bad = s < 0 || e < s || e > p.T;
      if (bad && lane == 0) flag_status(p.status, RL_DEV_BAD_OFFSETS);
      const bool longer = !bad && e - s > kWarpTokens;
      if (lane == 0) {
        span[warp][0] = s;
        span[warp][1] = longer ? e : s;
      }
      if (!bad && !longer) gae_trajectory<1>(p, i, s, e, nullptr, nullptr);
    }
    __syncthreads();
    for (int w = 0; w < here; ++w)
      if (span[w][1] > span[w][0])
        gae_trajectory<kWarps>(p, static_cast<int32_t>(base) + w, span[w][0], span[w][1], sh, sh_any);
    __syncthreads();  // span is rewritten for the next trajectories
  }
}

struct ValueArgs {
  int64_t rows;
  const float* values;
  const float* returns;
  const uint8_t* mask;
  const int32_t* token_traj;
  int32_t n_traj;
  const float* coef;
  float* d_values;
  double* row_loss;
  double* loss_accum;
  uint32_t* done;  // finished-CTA count in the workspace header
  int32_t* status;
};

// Each CTA adds its rows' terms in a fixed order (thread-strided, then warp and CTA) and leaves
// one partial per CTA in row_loss[blockIdx.x]; the last CTA to finish (a counter in the
// workspace header, which it resets) adds the partials in a fixed order into loss_accum.
//
// The FP64 pipe (16 clocks per warp instruction and SM) and the chain mask -> owner -> coefficient
// bound it, not the 21 bytes per row: so the floats are widened by integer instructions (one DFMA
// per row of four FP64 instructions), the grid is at most 4 CTAs per SM (the per-CTA sums are
// FP64 too), and VEC = 4 (every array on 16-byte boundaries, the mask on 4) takes four rows per
// thread and load.
template <int VEC>
__global__ void __launch_bounds__(256) value_loss_kernel(const ValueArgs p) {
  __shared__ double part[8];
  __shared__ uint32_t last;
  double acc = 0.0;
  // the value-loss terms of N rows whose inputs are in registers; the gradient goes to g
  auto terms = [&](auto n, const uint8_t* m, const int32_t* who, const float* v, const float* ret, float* g) {
    constexpr int N = decltype(n)::value;
    float c[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const bool in = who[k] >= 0 && who[k] < p.n_traj;
      if (m[k] != 0 && !in) flag_status(p.status, RL_DEV_BAD_TRAJ);
      c[k] = (m[k] != 0 && in) ? p.coef[who[k]] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const float d = v[k] - ret[k];
      const float cd = c[k] * d;
      g[k] = c[k] != 0.f ? 2.f * cd : 0.f;
      if (c[k] != 0.f) acc = fma(widen(cd), widen(d), acc);
    }
  };
  const int64_t first = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t vecs = VEC == 4 ? p.rows / 4 : 0;
  for (int64_t k = first; k < vecs; k += stride) {
    const uchar4 m = reinterpret_cast<const uchar4*>(p.mask)[k];
    const int4 w = reinterpret_cast<const int4*>(p.token_traj)[k];
    const float4 v = reinterpret_cast<const float4*>(p.values)[k], r = reinterpret_cast<const float4*>(p.returns)[k];
    const uint8_t ms[4] = {m.x, m.y, m.z, m.w};
    const int32_t who[4] = {w.x, w.y, w.z, w.w};
    const float vs[4] = {v.x, v.y, v.z, v.w}, rs[4] = {r.x, r.y, r.z, r.w};
    float g[4];
    terms(std::integral_constant<int, 4>{}, ms, who, vs, rs, g);
    reinterpret_cast<float4*>(p.d_values)[k] = make_float4(g[0], g[1], g[2], g[3]);
  }
  for (int64_t t = vecs * 4 + first; t < p.rows; t += stride) {
    const uint8_t m = p.mask[t];
    const int32_t who = p.token_traj[t];
    const float v = p.values[t], r = p.returns[t];
    float g;
    terms(std::integral_constant<int, 1>{}, &m, &who, &v, &r, &g);
    p.d_values[t] = g;
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += part[w];
    p.row_loss[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(p.done, 1u) == gridDim.x - 1 ? 1u : 0u;
    if (last) __threadfence();
  }
  __syncthreads();
  if (last) {  // uniform across the CTA
    double t = 0.0;
    for (uint32_t k = threadIdx.x; k < gridDim.x; k += blockDim.x) t += __ldcg(p.row_loss + k);
    t = warp_sum(t);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
      double u = 0.0;
      for (int w = 0; w < 8; ++w) u += part[w];
      *p.loss_accum += u;
      *p.done = 0u;
    }
  }
}

// A_t = R_{i(t)} - V_t and G_t = R_{i(t)} on trainable tokens, 0 elsewhere (any token order).
__global__ void __launch_bounds__(256) rollout_adv_kernel(int64_t T, const int32_t* __restrict__ token_traj,
                                                          const uint8_t* __restrict__ mask,
                                                          const float* __restrict__ values,
                                                          const float* __restrict__ rewards, int32_t n_traj,
                                                          float* __restrict__ adv, float* __restrict__ ret,
                                                          int32_t* status) {
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < T;
       t += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    float a = 0.f, g = 0.f;
    if (mask[t] != 0) {
      const int32_t i = token_traj[t];
      if (i < 0 || i >= n_traj) {
        flag_status(status, RL_DEV_BAD_TRAJ);
      } else {
        g = rewards[i];
        a = g - values[t];
      }
    }
    adv[t] = a;
    if (ret) ret[t] = g;
  }
}

static int grid_for(int64_t work, int per_block, int cap) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  return static_cast<int>(g < cap ? g : cap);
}

}  // namespace ppo
}  // namespace rl

extern "C" rl_status rl_masked_gae(int32_t n_traj, const int64_t* traj_offsets, int64_t n_tokens, const uint8_t* mask,
                                   const float* values, const float* token_rewards, const float* traj_rewards,
                                   float gamma, float gae_lambda, int32_t skip_masked, float* adv_out,
                                   float* returns_out, void* ws, size_t ws_bytes, rl_stream_t stream) {
  using namespace rl;
  clear_error();
  if (n_traj < 0 || n_tokens < 0) return set_error(RL_ERR_INVALID_ARG, "rl_masked_gae: negative size");
  if (!(gamma >= 0.f && gamma <= 1.f) || !(gae_lambda >= 0.f && gae_lambda <= 1.f))
    return set_error(RL_ERR_INVALID_ARG, "rl_masked_gae: gamma and lambda must lie in [0, 1]");
  if (skip_masked != 0 && skip_masked != 1)
    return set_error(RL_ERR_INVALID_ARG, "rl_masked_gae: skip_masked must be 0 or 1");
  if (!ws) return set_error(RL_ERR_INVALID_ARG, "rl_masked_gae: NULL workspace");
  if (ws_bytes < kWsHeader) return set_error(RL_ERR_WORKSPACE_TOO_SMALL, "rl_masked_gae: workspace too small");
  if (n_traj == 0) return RL_OK;
  if (!traj_offsets || (n_tokens > 0 && (!mask || !values || !adv_out)))
    return set_error(RL_ERR_INVALID_ARG, "rl_masked_gae: NULL array argument");
  ppo::GaeArgs a = {};
  a.n_traj = n_traj;
  a.offs = traj_offsets;
  a.T = n_tokens;
  a.mask = mask;
  a.values = values;
  a.token_rewards = token_rewards;
  a.traj_rewards = traj_rewards;
  a.gamma = gamma;
  a.lam = gae_lambda;
  a.skip = skip_masked;
  a.adv = adv_out;
  a.ret = returns_out;
  a.status = reinterpret_cast<int32_t*>(ws);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // a CTA (8 fit on an SM) per trajectory while they last, then up to a warp per trajectory
  const int grid = ppo::grid_for(n_traj, 1, 152 * 8);
  a.per_cta = std::min<int>(ppo::kWarps, (n_traj + grid - 1) / grid);
  ppo::gae_kernel<<<ppo::grid_for(n_traj, a.per_cta, 152 * 8), ppo::kThreads, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, "gae_kernel launch");
  return RL_OK;
}

extern "C" rl_status rl_value_loss_fwd_bwd(int64_t rows, const float* values, const float* returns,
                                           const uint8_t* mask, const int32_t* token_traj, int32_t n_traj,
                                           const float* coef, float* d_values, double* loss_accum, void* ws,
                                           size_t ws_bytes, rl_stream_t stream) {
  using namespace rl;
  clear_error();
  if (rows < 0 || n_traj < 0) return set_error(RL_ERR_INVALID_ARG, "rl_value_loss_fwd_bwd: negative size");
  if (!ws || !loss_accum) return set_error(RL_ERR_INVALID_ARG, "rl_value_loss_fwd_bwd: NULL argument");
  if (ws_bytes < kWsHeader + static_cast<size_t>(rows) * sizeof(double))
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL,
                     "rl_value_loss_fwd_bwd: workspace smaller than rl_workspace_size(rows, 0, 0)");
  if (rows == 0) return RL_OK;
  if (!values || !returns || !mask || !token_traj || !d_values || (n_traj > 0 && !coef))
    return set_error(RL_ERR_INVALID_ARG, "rl_value_loss_fwd_bwd: NULL array argument");
  ppo::ValueArgs a = {};
  a.rows = rows;
  a.values = values;
  a.returns = returns;
  a.mask = mask;
  a.token_traj = token_traj;
  a.n_traj = n_traj;
  a.coef = coef;
  a.d_values = d_values;
  double* row_loss = reinterpret_cast<double*>(static_cast<char*>(ws) + ws_row_loss_offset());
  a.row_loss = row_loss;
  a.loss_accum = loss_accum;
  a.done = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) + kWsValueDoneOffset);
  a.status = reinterpret_cast<int32_t*>(ws);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  auto on = [](const void* q, uintptr_t n) { return reinterpret_cast<uintptr_t>(q) % n == 0; };
  const bool vec = on(values, 16) && on(returns, 16) && on(token_traj, 16) && on(d_values, 16) && on(mask, 4);
  // at least one row per CTA, so that one partial per CTA fits the workspace
  const int blocks = ppo::grid_for(rows, vec ? 1024 : 256, 152 * 4);
  if (vec) ppo::value_loss_kernel<4><<<blocks, 256, 0, s>>>(a);
  else ppo::value_loss_kernel<1><<<blocks, 256, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, "value_loss_kernel launch");
  return RL_OK;  // the kernel's last CTA has added the loss into loss_accum
}

extern "C" rl_status rl_rollout_value_advantages(int64_t n_tokens, const int32_t* token_traj, const uint8_t* mask,
                                                 const float* values, const float* rewards, int32_t n_traj,
                                                 float* adv_out, float* returns_out, void* ws, size_t ws_bytes,
                                                 rl_stream_t stream) {
  using namespace rl;
  clear_error();
  if (n_tokens < 0 || n_traj < 0) return set_error(RL_ERR_INVALID_ARG, "rl_rollout_value_advantages: negative size");
  if (!ws) return set_error(RL_ERR_INVALID_ARG, "rl_rollout_value_advantages: NULL workspace");
  if (ws_bytes < kWsHeader)
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL, "rl_rollout_value_advantages: workspace too small");
  if (n_tokens == 0) return RL_OK;
  if (!token_traj || !mask || !values || !adv_out || (n_traj > 0 && !rewards))
    return set_error(RL_ERR_INVALID_ARG, "rl_rollout_value_advantages: NULL array argument");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  ppo::rollout_adv_kernel<<<ppo::grid_for(n_tokens, 256, 152 * 8), 256, 0, s>>>(
      n_tokens, token_traj, mask, values, rewards, n_traj, adv_out, returns_out, reinterpret_cast<int32_t*>(ws));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, "rollout_adv_kernel launch");
  return RL_OK;
}
