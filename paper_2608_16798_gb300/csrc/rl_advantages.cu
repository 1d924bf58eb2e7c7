// Group-relative advantages and loss coefficients over ragged trajectories.
//
//   count_adv_kernel    one launch, two kinds of CTA: the first count L_i, the
//                       trainable tokens of each trajectory (a CTA or a warp
//                       per trajectory span, writing token_traj[t] = i; or, by owner,
//                       a grid-stride pass over tokens in any order), the 1 /
//                       sum_t M_{i,t} normaliser of the masked GRPO objective
//                       (Sec. 2.3.2); the others form A_i = (R_i - mu_g) /
//                       (sigma_g + eps) per group (a segment of a warp per group:
//                       mean and population standard deviation of the valid
//                       members' rewards in double precision; Sec. 2.3.2 GRPO advantage,
//                       Sec. 3.2.3; discarded rollouts leave the statistics and
//                       get A = 0, Sec. 3.4). Counts and advantages do not depend
//                       on each other.
//   coef_kernel         N = #{valid i : L_i > 0} and S = sum of their L_i (every
//                       CTA forms both, integer sums, so any order gives the same
//                       values), then c_i for its share of the trajectories, and
//                       A = 0 for trajectories outside every group.
//
// Every kind of work is spread over the GPU: a batch of many small groups (4,096
// groups of 4) costs no more than a few large ones. Both kernels are
// latency-bound: they touch ~T + 30 n bytes, well under 0.1% of the logits
// stream of one microbatch.
#include <cstdint>

#include "rl_device.cuh"
#include "rl_host.h"

namespace rl {

constexpr int kAdvThreads = 256;
constexpr int kAdvWarps = kAdvThreads / 32;

// Trainable tokens of [s, e) and the owner i of each token of it, by the `n` threads of which this
// is thread k (a few lanes, a warp or a CTA): 16 mask bytes a load and four owners a store over the part of the span whose
// addresses are 16-byte aligned (a warp per span with one byte and one owner at a time took 14 us
// for 512 spans of 512 to 8,192 tokens, a chain of 256 trips of the longest one), one token at a
// time over the rest.
__device__ __forceinline__ int32_t count_span(int64_t i, int k, int n, int64_t s, int64_t e, const uint8_t* mask,
                                              int32_t* token_traj_out) {
  int32_t cnt = 0;
  int64_t v0 = e, v1 = e;  // vector part
  if (e - s >= 64) {
    v0 = s + ((16 - (reinterpret_cast<uintptr_t>(mask + s) & 15)) & 15);
    if (token_traj_out && (reinterpret_cast<uintptr_t>(token_traj_out + v0) & 15) != 0) v0 = e;
    v1 = v0 + (e - v0) / 16 * 16;
  }
  const int32_t who = static_cast<int32_t>(i);
#pragma unroll 4
  for (int64_t t = v0 + static_cast<int64_t>(k) * 16; t < v1; t += static_cast<int64_t>(n) * 16) {
    const uint4 w = *reinterpret_cast<const uint4*>(mask + t);
    cnt += __popc(__vsetne4(w.x, 0u)) + __popc(__vsetne4(w.y, 0u)) + __popc(__vsetne4(w.z, 0u)) +
           __popc(__vsetne4(w.w, 0u));
  }
  if (token_traj_out)
    for (int64_t t = v0 + static_cast<int64_t>(k) * 4; t < v1; t += static_cast<int64_t>(n) * 4)
      *reinterpret_cast<int4*>(token_traj_out + t) = make_int4(who, who, who, who);
  auto one = [&](int64_t t) {
    cnt += mask[t] != 0;
    if (token_traj_out) token_traj_out[t] = who;
  };
  const int64_t h1 = v0 < v1 ? v0 : e;  // tokens before the vector part, or all of them
  for (int64_t t = s + k; t < h1; t += n) one(t);
  if (v0 < v1)
    for (int64_t t = v1 + k; t < e; t += n) one(t);
  return cnt;
}

// L_i by owner, for tokens in any order (tree-packed batches, Sec. 3.2.3: each shared prefix
// token is one token of its rollout): lanes of a warp with the same owner are counted together
// and one integer atomic per owner and warp adds them (the counts are exact in any order).
// Warp w of `warps` takes the 32-token runs w, w + warps, ... (n_tok_out zeroed before).
__device__ __forceinline__ void count_owners(int64_t w, int64_t warps, int lane, int64_t n_tokens,
                                             const int32_t* token_traj, const uint8_t* mask, int32_t n_traj,
                                             int32_t* n_tok_out, int32_t* status) {
  for (int64_t base = w * 32; base < n_tokens; base += warps * 32) {
    const int64_t t = base + lane;
    int32_t who = -1;
    if (t < n_tokens && mask[t] != 0) {
      const int32_t i = token_traj[t];
      if (i < 0 || i >= n_traj) flag_status(status, RL_DEV_BAD_TRAJ);
      else who = i;
    }
    const unsigned peers = __match_any_sync(0xffffffffu, who);
    if (who >= 0 && lane == __ffs(peers) - 1) atomicAdd(&n_tok_out[who], __popc(peers));
  }
}

// A_i for the members of group g (one warp): mean and population standard deviation of the
// valid members' rewards in double precision, each A_i rounded once to float. Invalid members,
// and every member of a group with no valid member or whose valid rewards are all equal, get 0.
__device__ __forceinline__ void group_advantage(int64_t g, int lane, int32_t n_traj, const int32_t* group_offsets,
                                                const float* rewards, const uint8_t* traj_valid, double adv_eps,
                                                float* adv_out, int32_t* status) {
  const int b = group_offsets[g], e = group_offsets[g + 1];
  if (b < 0 || e < b || e > n_traj) {
    if (lane == 0) flag_status(status, RL_DEV_BAD_OFFSETS);
    return;
  }
  // pass 1: count, sum, and min / max (all-equal test) over valid members
  int k = 0;
  double sum = 0.0;
  float lo = __int_as_float(0x7f800000), hi = -__int_as_float(0x7f800000);
  for (int i = b + lane; i < e; i += 32) {
    if (traj_valid && traj_valid[i] == 0) continue;
    const float r = rewards[i];
    ++k;
    sum += static_cast<double>(r);
    lo = fminf(lo, r);
    hi = fmaxf(hi, r);
  }
  k = warp_sum(k);
  sum = warp_sum(sum);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (k == 0 || lo == hi) {  // nothing valid, or all valid rewards equal: A = 0
    for (int i = b + lane; i < e; i += 32) adv_out[i] = 0.f;
    return;
  }
  const double mu = sum / k;
  double sq = 0.0;
  for (int i = b + lane; i < e; i += 32) {
    if (traj_valid && traj_valid[i] == 0) continue;
    const double d = static_cast<double>(rewards[i]) - mu;
    sq += d * d;
  }
  sq = warp_sum(sq);
  const double denom = sqrt(sq / k) + adv_eps;
  for (int i = b + lane; i < e; i += 32) {
    const bool valid = !traj_valid || traj_valid[i] != 0;
    adv_out[i] = valid ? static_cast<float>((static_cast<double>(rewards[i]) - mu) / denom) : 0.f;
  }
}

// A_i for 32 / W neighbouring groups by one warp, a segment of W lanes each (W a power of two, at
// least the batch's mean group size): the FP64 pipe bounds this (two lanes per clock and SM, the
// same for one active lane of a warp as for 32), so a warp per group of 4 spent an eighth of it;
// 4,096 groups of 4 took 27 us with the counts. Sums go over the same lanes in the same butterfly
// order as in group_advantage (whose higher lanes add zeros), so a group of at most W members
// gets the same bits. Groups of more than 8 W members are left to the whole warp.
__device__ __forceinline__ void group_advantages(int64_t g0, int W, int lane, int32_t n_traj, int32_t n_groups,
                                                 const int32_t* group_offsets, const float* rewards,
                                                 const uint8_t* traj_valid, double adv_eps, float* adv_out,
                                                 int32_t* status) {
  const int64_t g = g0 + lane / W;
  const int sl = lane % W;
  int b = 0, e = 0;
  if (g < n_groups) {
    b = group_offsets[g];
    e = group_offsets[g + 1];
    if (b < 0 || e < b || e > n_traj) {
      if (sl == 0) flag_status(status, RL_DEV_BAD_OFFSETS);
      b = e = 0;
    }
  }
  unsigned big = __ballot_sync(0xffffffffu, sl == 0 && e - b > 8 * W);
  if (e - b > 8 * W) e = b;
  int k = 0;
  double sum = 0.0;
  float lo = __int_as_float(0x7f800000), hi = -__int_as_float(0x7f800000);
  for (int i = b + sl; i < e; i += W) {
    if (traj_valid && traj_valid[i] == 0) continue;
    const float r = rewards[i];
    ++k;
    sum += static_cast<double>(r);
    lo = fminf(lo, r);
    hi = fmaxf(hi, r);
  }
  __syncwarp();
  for (int o = W / 2; o > 0; o >>= 1) {
    k += __shfl_xor_sync(0xffffffffu, k, o);
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  const bool zero = k == 0 || lo == hi;  // nothing valid, or all valid rewards equal: A = 0
  const double mu = sum / (k > 0 ? k : 1);
  double sq = 0.0;
  for (int i = b + sl; i < e && !zero; i += W) {
    if (traj_valid && traj_valid[i] == 0) continue;
    const double d = static_cast<double>(rewards[i]) - mu;
    sq += d * d;
  }
  __syncwarp();
  for (int o = W / 2; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  const double denom = sqrt(sq / (k > 0 ? k : 1)) + adv_eps;
  for (int i = b + sl; i < e; i += W) {
    const bool valid = !zero && (!traj_valid || traj_valid[i] != 0);
    adv_out[i] = valid ? static_cast<float>((static_cast<double>(rewards[i]) - mu) / denom) : 0.f;
  }
  __syncwarp();
  for (; big; big &= big - 1)
    group_advantage(g0 + (__ffs(big) - 1) / W, lane, n_traj, group_offsets, rewards, traj_valid, adv_eps, adv_out,
                    status);
}

struct CountAdvArgs {
  int32_t n_traj, n_groups;
  int64_t n_tokens;
  int64_t count_blocks, adv_blocks;  // CTAs [0, adv_blocks) form advantages, the rest count
  int32_t span_threads;              // threads that count a span: 8 lanes, a warp, or the whole CTA
  int32_t seg;                     // lanes per group
  const int64_t* traj_offsets;     // spans (rl_group_advantages)
  const int32_t* token_traj;       // owners (rl_group_advantages_by_owner)
  const uint8_t* mask;
  const int32_t* group_offsets;
  const float* rewards;
  const uint8_t* traj_valid;
  double adv_eps;
  float* adv_out;
  float* coef_out;
  int32_t* n_tok_out;
  int32_t* token_traj_out;
  int32_t* status;
};

template <bool BY_OWNER>
__global__ void __launch_bounds__(kAdvThreads) count_adv_kernel(const CountAdvArgs a) {
  __shared__ int32_t part[kAdvWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // the advantages first: theirs is the longer chain (two trips to memory, then FP64 divisions and
  // a square root)
  const int64_t block = static_cast<int64_t>(blockIdx.x) - a.adv_blocks;
  if (block >= 0) {
    if (BY_OWNER) {
      count_owners(block * kAdvWarps + warp, a.count_blocks * kAdvWarps, lane, a.n_tokens, a.token_traj, a.mask,
                   a.n_traj, a.n_tok_out, a.status);
      return;
    }
    const int n = a.span_threads;
    const int k = static_cast<int>(threadIdx.x) % n;  // this thread within its span's threads
    const int64_t i = block * (kAdvThreads / n) + threadIdx.x / n;
    int32_t cnt = 0;
    if (i < a.n_traj) {
      const int64_t s = a.traj_offsets[i], e = a.traj_offsets[i + 1];
      const bool bad = s < 0 || e < s || e > a.n_tokens;
      if (bad && k == 0) flag_status(a.status, RL_DEV_BAD_OFFSETS);
      if (!bad) cnt = count_span(i, k, n, s, e, a.mask, a.token_traj_out);
    }
    __syncwarp();
    for (int o = (n < 32 ? n : 32) / 2; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    if (n > 32) {
      if (lane == 0) part[warp] = cnt;
      __syncthreads();
      cnt = 0;
      for (int w = 0; w < kAdvWarps; ++w) cnt += part[w];
    }
    if (k == 0 && i < a.n_traj) a.n_tok_out[i] = cnt;
  } else {
    const int per = 32 / a.seg;  // groups of a warp
    const int64_t g0 = (static_cast<int64_t>(blockIdx.x) * kAdvWarps + warp) * per;
    if (g0 < a.n_groups)
      group_advantages(g0, a.seg, lane, a.n_traj, a.n_groups, a.group_offsets, a.rewards, a.traj_valid, a.adv_eps,
                       a.adv_out, a.status);
  }
}

// Coefficients c_i (Sec. 2.3.2: 1 / (N L_i) under seq-mean-token-mean; 1 / S under token-mean;
// 1 under token-sum) for valid trajectories with L_i > 0, else 0; A = 0 for trajectories
// before the first group or after the last.
__global__ void __launch_bounds__(kAdvThreads) coef_kernel(int32_t n_traj, int32_t n_groups,
                                                           const int32_t* __restrict__ group_offsets,
                                                           const uint8_t* __restrict__ traj_valid,
                                                           const int32_t* __restrict__ n_tok, int32_t loss_agg,
                                                           float* __restrict__ adv_out, float* __restrict__ coef_out) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ long long red_n[kAdvWarps], red_s[kAdvWarps];
  long long cnt = 0, tok = 0;
  // 16 loads in flight: at 16,384 trajectories a thread's 64 counts are 4 trips to L2, not 16
#pragma unroll 16
  for (int i = tid; i < n_traj; i += kAdvThreads) {
    const int32_t L = n_tok[i];
    const bool counted = (!traj_valid || traj_valid[i] != 0) && L > 0;
    cnt += counted;
    tok += counted ? L : 0;
  }
  cnt = warp_sum(cnt);
  tok = warp_sum(tok);
  if (lane == 0) {
    red_n[warp] = cnt;
    red_s[warp] = tok;
  }
  __syncthreads();
  long long N = 0, S = 0;
  for (int w = 0; w < kAdvWarps; ++w) {
    N += red_n[w];
    S += red_s[w];
  }
  int32_t first = n_traj, last = n_traj;  // trajectories [first, last) belong to groups
  if (n_groups > 0) {
    first = min(max(group_offsets[0], 0), n_traj);
    last = min(max(group_offsets[n_groups], first), n_traj);
  }
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * kAdvThreads + tid; i < n_traj;
       i += static_cast<int64_t>(gridDim.x) * kAdvThreads) {
    if (i < first || i >= last) adv_out[i] = 0.f;
    const int32_t L = n_tok[i];
    const bool counted = (!traj_valid || traj_valid[i] != 0) && L > 0;
    float c = 0.f;
    if (counted) {
      if (loss_agg == RL_AGG_SEQ_MEAN_TOKEN_MEAN)
        c = static_cast<float>(1.0 / (static_cast<double>(N) * static_cast<double>(L)));
      else if (loss_agg == RL_AGG_TOKEN_MEAN)
        c = static_cast<float>(1.0 / static_cast<double>(S));
      else
        c = 1.f;
    }
    coef_out[i] = c;
  }
}

// Launches count_adv_kernel (count_blocks counting CTAs, then one warp per group) and
// coef_kernel on stream s.
template <bool BY_OWNER>
static rl_status launch_advantages(CountAdvArgs a, int64_t count_blocks, const rl_loss_params* params, const char* fn,
                                   cudaStream_t s) {
  a.count_blocks = count_blocks;
  // lanes per group: the power of two at or above the mean group size
  const int64_t mean = a.n_groups > 0 ? (static_cast<int64_t>(a.n_traj) + a.n_groups - 1) / a.n_groups : 32;
  a.seg = 2;
  while (a.seg < mean && a.seg < 32) a.seg *= 2;
  const int64_t per_cta = static_cast<int64_t>(kAdvWarps) * (32 / a.seg);
  a.adv_blocks = (a.n_groups + per_cta - 1) / per_cta;
  const int64_t blocks = count_blocks + a.adv_blocks;
  if (blocks > 0) {
    count_adv_kernel<BY_OWNER><<<static_cast<unsigned>(blocks), kAdvThreads, 0, s>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, (std::string(fn) + ": count_adv_kernel launch").c_str());
  }
  // every CTA reads all n_tok once for N and S: a few CTAs per wave of the GPU at most
  int64_t cb = (static_cast<int64_t>(a.n_traj) + kAdvThreads - 1) / kAdvThreads;
  if (cb > 152) cb = 152;
  coef_kernel<<<static_cast<unsigned>(cb), kAdvThreads, 0, s>>>(a.n_traj, a.n_groups, a.group_offsets, a.traj_valid,
                                                                 a.n_tok_out, params->loss_agg, a.adv_out, a.coef_out);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, (std::string(fn) + ": coef_kernel launch").c_str());
  return RL_OK;
}

}  // namespace rl

extern "C" rl_status rl_group_advantages(int32_t n_traj, int32_t n_groups, const int32_t* group_offsets,
                                         const float* rewards, const uint8_t* traj_valid, int64_t n_tokens,
                                         const int64_t* traj_offsets, const uint8_t* mask,
                                         const rl_loss_params* params, float* adv_out, float* coef_out,
                                         int32_t* n_tok_out, int32_t* token_traj_out, void* ws,
                                         size_t ws_bytes, rl_stream_t stream) {
  using namespace rl;
  clear_error();
  if (n_traj < 0 || n_groups < 0 || n_tokens < 0)
    return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: negative size");
  if (!params) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: params is NULL");
  if (!ws) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: ws is NULL");
  if (ws_bytes < rl_workspace_size(0, 0, 0))
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL, "rl_group_advantages: workspace too small");
  if (params->loss_agg < RL_AGG_SEQ_MEAN_TOKEN_MEAN || params->loss_agg > RL_AGG_TOKEN_SUM)
    return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: unknown loss_agg");
  if (!(params->adv_eps >= 0.f)) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: adv_eps < 0");
  if (n_traj == 0) return RL_OK;
  if (!group_offsets && n_groups > 0) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: group_offsets is NULL");
  if (!rewards || !traj_offsets || !adv_out || !coef_out || !n_tok_out)
    return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: NULL array argument");
  if (n_tokens > 0 && !mask) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages: mask is NULL");
  if (n_tokens > INT32_MAX) return set_error(RL_ERR_UNSUPPORTED, "rl_group_advantages: more than 2^31 - 1 tokens");
  CountAdvArgs a = {};
  a.n_traj = n_traj;
  a.n_groups = n_groups;
  a.n_tokens = n_tokens;
  a.traj_offsets = traj_offsets;
  a.mask = mask;
  a.group_offsets = group_offsets;
  a.rewards = rewards;
  a.traj_valid = traj_valid;
  a.adv_eps = static_cast<double>(params->adv_eps);
  a.adv_out = adv_out;
  a.coef_out = coef_out;
  a.n_tok_out = n_tok_out;
  a.token_traj_out = token_traj_out;
  a.status = reinterpret_cast<int32_t*>(ws);
  // a CTA per span while one wave of the GPU (8 CTAs per SM) holds them, else a warp per span, or 8
  // lanes where the mean span is below 64 tokens (16,384 spans of 8 tokens were 1.7 waves of warps)
  a.span_threads = n_traj <= 152 * 8 ? kAdvThreads : n_tokens >= 64 * static_cast<int64_t>(n_traj) ? 32 : 8;
  const int64_t per_cta = kAdvThreads / a.span_threads;
  const int64_t count_blocks = (n_traj + per_cta - 1) / per_cta;
  return launch_advantages<false>(a, count_blocks, params, "rl_group_advantages",
                                  reinterpret_cast<cudaStream_t>(stream));
}

extern "C" rl_status rl_group_advantages_by_owner(int32_t n_traj, int32_t n_groups, const int32_t* group_offsets,
                                                  const float* rewards, const uint8_t* traj_valid, int64_t n_tokens,
                                                  const int32_t* token_traj, const uint8_t* mask,
                                                  const rl_loss_params* params, float* adv_out, float* coef_out,
                                                  int32_t* n_tok_out, void* ws, size_t ws_bytes,
                                                  rl_stream_t stream) {
  using namespace rl;
  clear_error();
  if (n_traj < 0 || n_groups < 0 || n_tokens < 0)
    return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages_by_owner: negative size");
  if (!params) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages_by_owner: params is NULL");
  if (!ws) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages_by_owner: ws is NULL");
  if (ws_bytes < rl_workspace_size(0, 0, 0))
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL, "rl_group_advantages_by_owner: workspace too small");
  if (params->loss_agg < RL_AGG_SEQ_MEAN_TOKEN_MEAN || params->loss_agg > RL_AGG_TOKEN_SUM)
    return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages_by_owner: unknown loss_agg");
  if (!(params->adv_eps >= 0.f)) return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages_by_owner: adv_eps < 0");
  if (n_traj == 0) return RL_OK;
  if (!group_offsets && n_groups > 0)
    return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages_by_owner: group_offsets is NULL");
  if (!rewards || !adv_out || !coef_out || !n_tok_out || (n_tokens > 0 && (!token_traj || !mask)))
    return set_error(RL_ERR_INVALID_ARG, "rl_group_advantages_by_owner: NULL array argument");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemsetAsync(n_tok_out, 0, static_cast<size_t>(n_traj) * sizeof(int32_t), s);
  if (e != cudaSuccess) return cuda_error(e, "rl_group_advantages_by_owner: cudaMemsetAsync");
  CountAdvArgs a = {};
  a.n_traj = n_traj;
  a.n_groups = n_groups;
  a.n_tokens = n_tokens;
  a.token_traj = token_traj;
  a.mask = mask;
  a.group_offsets = group_offsets;
  a.rewards = rewards;
  a.traj_valid = traj_valid;
  a.adv_eps = static_cast<double>(params->adv_eps);
  a.adv_out = adv_out;
  a.coef_out = coef_out;
  a.n_tok_out = n_tok_out;
  a.status = reinterpret_cast<int32_t*>(ws);
  // grid-stride over 32-token runs: at most 8 CTAs per SM
  int64_t count_blocks = (n_tokens + kAdvThreads - 1) / kAdvThreads;
  if (count_blocks > 152 * 8) count_blocks = 152 * 8;
  return launch_advantages<true>(a, count_blocks, params, "rl_group_advantages_by_owner", s);
}
