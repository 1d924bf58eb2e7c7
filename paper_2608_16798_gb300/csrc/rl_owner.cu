// Sums over the tokens that a unit owns, for any token order: sequence-level importance
// weights (Sec. 3.2.4) over trajectories or over the deduplicated tokens of a rollout's
// prefix tree (Sec. 3.2.3), where a unit's tokens need not be contiguous.
//
//   owner_logratio_kernel  per token with M_t = 1: d = log pi_old - log pi_rollout, rounded to a
//                          fixed-point integer (2^-40 units) as the double difference would be;
//                          a lane takes four neighbouring tokens, the lanes of a warp with the
//                          same owner add theirs (runs of equal owners by a segmented scan, other
//                          orders by __match_any_sync), one 64-bit integer atomic per run or
//                          owner. Integer addition is associative, so the sums do not depend on
//                          the order of the atomics.
//   seq_weight_kernel      per unit: S = sum * 2^-40, w = min(exp(S), c-bar); optionally
//                          scales the unit's advantage by w.
//   token_scale_kernel     optionally scales per-token advantages by their owner's w.
#include <cstdint>

#include "rl_device.cuh"
#include "rl_host.h"

namespace rl {
namespace owner {

constexpr double kFix = 1099511627776.0;  // 2^40
constexpr double kMaxTerm = 4194304.0;    // |d| <= 2^22 per token keeps every sum inside int64

// x 2^40 for a float of magnitude 0 or in [2^-17, 2^12): a whole number, the float's last bit being
// worth at least 2^-40. e is the biased exponent.
__device__ __forceinline__ long long fixed40(uint32_t bits, uint32_t e) {
  const long long m = static_cast<long long>((bits & 0x7FFFFFu) | 0x800000u) << ((e - 110u) & 63u);
  const long long v = (bits << 1) == 0u ? 0 : m;
  return (bits >> 31) ? -v : v;
}

// round((old - roll) 2^40) with the difference taken in double. Where both are multiples of 2^-40
// below 2^12 the double difference is exact, and so is this integer one; the other values take the
// FP64 pipe (six instructions of 16 clocks each per warp, which bound the kernel when every token
// took them).
__device__ __forceinline__ long long log_ratio_fixed(float old, float roll, int32_t* status) {
  const uint32_t a = __float_as_uint(old), b = __float_as_uint(roll);
  const uint32_t ea = (a >> 23) & 0xFFu, eb = (b >> 23) & 0xFFu;
  if ((ea - 110u <= 28u || (a << 1) == 0u) && (eb - 110u <= 28u || (b << 1) == 0u))
    return fixed40(a, ea) - fixed40(b, eb);
  double d = static_cast<double>(old) - static_cast<double>(roll);
  if (!(fabs(d) <= kMaxTerm)) {
    flag_status(status, RL_DEV_BAD_VALUE);
    d = d != d ? 0.0 : (d > 0 ? kMaxTerm : -kMaxTerm);
  }
  return __double2ll_rn(d * kFix);
}

// Adds q of every lane to acc[who] (who < 0: nothing), one atomic per run of neighbouring lanes
// with the same owner while the warp has few runs, else one per owner.
__device__ __forceinline__ void add_by_owner(int32_t who, long long q, int lane, unsigned long long* acc) {
  const int32_t prev = __shfl_up_sync(0xffffffffu, who, 1);
  const unsigned heads = __ballot_sync(0xffffffffu, lane == 0 || who != prev);
  if (__popc(heads) <= 8) {
    const unsigned later = lane == 31 ? 0u : heads >> (lane + 1);
    const int end = later ? lane + __ffs(later) - 1 : 31;  // last lane of this lane's run
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const long long o = __shfl_down_sync(0xffffffffu, q, off);
      if (lane + off <= end) q += o;
    }
    if (who >= 0 && ((heads >> lane) & 1u)) atomicAdd(&acc[who], static_cast<unsigned long long>(q));
    return;
  }
  const unsigned peers = __match_any_sync(0xffffffffu, who);
  long long sum = 0;
#pragma unroll 4
  for (int j = 0; j < 32; ++j) {
    const long long v = __shfl_sync(0xffffffffu, q, j);
    if ((peers >> j) & 1u) sum += v;
  }
  if (who >= 0 && lane == __ffs(peers) - 1) atomicAdd(&acc[who], static_cast<unsigned long long>(sum));
}

// A warp takes 128 tokens at a time, a lane four neighbouring ones: by 16-byte loads with VEC
// (arrays on 16-byte boundaries, the mask on 4), else one by one.
template <bool VEC>
__global__ void __launch_bounds__(256) owner_logratio_kernel(int64_t T, const int32_t* __restrict__ token_traj,
                                                             const uint8_t* __restrict__ mask,
                                                             const float* __restrict__ old_logp,
                                                             const float* __restrict__ rollout_logp, int32_t n_traj,
                                                             unsigned long long* __restrict__ acc, int32_t* status) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x / 32);
  for (int64_t base = (static_cast<int64_t>(blockIdx.x) * (blockDim.x / 32) + (threadIdx.x >> 5)) * 128; base < T;
       base += warps * 128) {
    const int64_t t0 = base + lane * 4;
    uint8_t m[4];
    int32_t who[4];
    float old[4], roll[4];
    if (VEC && t0 + 4 <= T) {
      const uchar4 mv = *reinterpret_cast<const uchar4*>(mask + t0);
      const int4 wv = *reinterpret_cast<const int4*>(token_traj + t0);
      const float4 ov = *reinterpret_cast<const float4*>(old_logp + t0);
      const float4 rv = *reinterpret_cast<const float4*>(rollout_logp + t0);
      m[0] = mv.x; m[1] = mv.y; m[2] = mv.z; m[3] = mv.w;
      who[0] = wv.x; who[1] = wv.y; who[2] = wv.z; who[3] = wv.w;
      old[0] = ov.x; old[1] = ov.y; old[2] = ov.z; old[3] = ov.w;
      roll[0] = rv.x; roll[1] = rv.y; roll[2] = rv.z; roll[3] = rv.w;
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const bool in = t0 + k < T;
        m[k] = in ? mask[t0 + k] : 0;
        who[k] = in ? token_traj[t0 + k] : -1;
        old[k] = in ? old_logp[t0 + k] : 0.f;
        roll[k] = in ? rollout_logp[t0 + k] : 0.f;
      }
    }
    long long q[4], sum = 0;
    int32_t own = -1;  // the one owner of this lane's trained tokens ...
    bool one = true;   // ... if there is only one
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (m[k] != 0 && (who[k] < 0 || who[k] >= n_traj)) flag_status(status, RL_DEV_BAD_TRAJ);
      if (m[k] == 0 || who[k] < 0 || who[k] >= n_traj) who[k] = -1;
      q[k] = who[k] >= 0 ? log_ratio_fixed(old[k], roll[k], status) : 0;
      if (who[k] >= 0) {
        one = one && (own < 0 || own == who[k]);
        own = who[k];
      }
      sum += q[k];
    }
    if (__all_sync(0xffffffffu, one)) {
      add_by_owner(own, sum, lane, acc);
    } else {
#pragma unroll 1
      for (int k = 0; k < 4; ++k) {
        const int32_t w = k == 0 ? who[0] : k == 1 ? who[1] : k == 2 ? who[2] : who[3];
        const long long v = k == 0 ? q[0] : k == 1 ? q[1] : k == 2 ? q[2] : q[3];
        add_by_owner(w, v, lane, acc);
      }
    }
  }
}

__global__ void __launch_bounds__(256) seq_weight_kernel(int32_t n_traj, const unsigned long long* __restrict__ acc,
                                                         float cap, float* __restrict__ weight_out,
                                                         float* __restrict__ log_ratio_out,
                                                         float* __restrict__ traj_adv) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_traj) return;
  const double S = static_cast<double>(static_cast<long long>(acc[i])) / kFix;
  double w = exp(S);
  if (cap > 0.f && w > cap) w = cap;
  const float wf = static_cast<float>(w);
  weight_out[i] = wf;
  if (log_ratio_out) log_ratio_out[i] = static_cast<float>(S);
  if (traj_adv) traj_adv[i] *= wf;
}

__global__ void __launch_bounds__(256) token_scale_kernel(int64_t T, const int32_t* __restrict__ token_traj,
                                                          int32_t n_traj, const float* __restrict__ weight,
                                                          float* __restrict__ token_adv) {
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  for (int64_t t = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; t < T; t += stride) {
    const int32_t i = token_traj[t];
    if (i >= 0 && i < n_traj) token_adv[t] *= weight[i];
  }
}

static int grid_for(int64_t work, int per_block, int cap) {
  int64_t g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  return static_cast<int>(g < cap ? g : cap);
}

}  // namespace owner
}  // namespace rl

extern "C" rl_status rl_sequence_is_weights(int32_t n_traj, int64_t n_tokens, const int32_t* token_traj,
                                            const uint8_t* mask, const float* old_logp, const float* rollout_logp,
                                            float cap, float* weight_out, float* log_ratio_out,
                                            float* traj_adv_inout, float* token_adv_inout, void* ws, size_t ws_bytes,
                                            rl_stream_t stream) {
  using namespace rl;
  clear_error();
  if (n_traj < 0 || n_tokens < 0) return set_error(RL_ERR_INVALID_ARG, "rl_sequence_is_weights: negative size");
  if (cap != cap) return set_error(RL_ERR_INVALID_ARG, "rl_sequence_is_weights: cap is NaN");
  if (!ws) return set_error(RL_ERR_INVALID_ARG, "rl_sequence_is_weights: NULL workspace");
  if (ws_bytes < kWsHeader + static_cast<size_t>(n_traj) * sizeof(unsigned long long))
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL,
                     "rl_sequence_is_weights: workspace smaller than rl_workspace_size(n_traj, 0, 0)");
  if (n_traj == 0) return RL_OK;
  if (!weight_out || (n_tokens > 0 && (!token_traj || !mask || !old_logp || !rollout_logp)))
    return set_error(RL_ERR_INVALID_ARG, "rl_sequence_is_weights: NULL array argument");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  int32_t* status = reinterpret_cast<int32_t*>(ws);
  unsigned long long* acc =
      reinterpret_cast<unsigned long long*>(static_cast<char*>(ws) + ws_row_loss_offset());
  cudaError_t e = cudaMemsetAsync(acc, 0, static_cast<size_t>(n_traj) * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return cuda_error(e, "cudaMemsetAsync");
  if (n_tokens > 0) {
    auto on = [](const void* q, uintptr_t n) { return reinterpret_cast<uintptr_t>(q) % n == 0; };
    const bool vec = on(token_traj, 16) && on(old_logp, 16) && on(rollout_logp, 16) && on(mask, 4);
    auto kern = vec ? owner::owner_logratio_kernel<true> : owner::owner_logratio_kernel<false>;
    kern<<<owner::grid_for(n_tokens, 1024, 152 * 8), 256, 0, s>>>(n_tokens, token_traj, mask, old_logp, rollout_logp,
                                                                  n_traj, acc, status);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "owner_logratio_kernel launch");
  }
  owner::seq_weight_kernel<<<(n_traj + 255) / 256, 256, 0, s>>>(n_traj, acc, cap, weight_out, log_ratio_out,
                                                                 traj_adv_inout);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_error(e, "seq_weight_kernel launch");
  if (token_adv_inout && n_tokens > 0) {
    owner::token_scale_kernel<<<owner::grid_for(n_tokens, 256, 152 * 8), 256, 0, s>>>(n_tokens, token_traj, n_traj,
                                                                                      weight_out, token_adv_inout);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "token_scale_kernel launch");
  }
  return RL_OK;
}
