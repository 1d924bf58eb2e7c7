// Fixed-order reductions: batch summaries of the per-token statistics that
// rl_policy_loss_fwd_bwd and rl_fused_head_loss_fwd_bwd write: the number of trained tokens, of clipped ones, and the
// sums of entropy, KL and ratio over them (the clip fraction and the mean policy entropy that
// are tracked during training, Sec. 4). Fixed assignment of rows to threads and a fixed
// reduction order in double precision: the sums are the same on every run.
#include <algorithm>
#include <cstdint>
#include <map>
#include <mutex>

#include "rl_device.cuh"
#include "rl_host.h"

namespace rl {

// Batch summary of the per-token statistics: up to kSumSlots clusters of kSumCluster CTAs (one
// launch). Global thread g takes rows g, g + G, g + 2G, ... (G = all threads) in groups of
// kSumUnroll rows whose loads are issued together (mask and owner, then the coefficients, then the
// statistics: three dependent round trips per group instead of per row); each thread adds its
// rows in order, then the warps, the CTA and the cluster's CTAs are combined in a fixed order (the
// CTA totals meet in rank 0's shared memory), and the last cluster to finish adds the clusters'
// totals in order: the grid depends on the row count alone, so the sums are the same on every run.
//
// What bounded one cluster of 8 was the FP64 pipe (two lanes per clock and SM: 16 clocks per warp
// instruction): ten such instructions per row. So the number of rows and of clipped ones (a flag of 1)
// are counted in integers, the floats are widened by integer instructions, and three DADD per row remain;
// and the rows spread over up to 80 SMs. The slots that hold a cluster's five totals are spare bytes of
// the 256-byte workspace header, which every caller has: five of them fit, which with clusters of 16
// gives 80 CTAs. 1.42 M rows: 487 -> 30 us, 131,072 rows: 56 -> 17. What bounds it now is latency (the
// three dependent trips, four scalar loads of each 20-byte row, the cluster's launch and barriers): sums in
// 64-bit integers, without any FP64 per row, took as long.
constexpr int kSumThreads = 1024;
constexpr int kSumCluster = 16;  // 8 where the device has no room for one of 16
constexpr int kSumUnroll = 4;
constexpr int kSumSlots = 5;
static_assert(kWsSummaryOffset + kSumSlots * 5 * sizeof(double) <= kWsHeader, "summary slots fit the header");

__device__ __forceinline__ void st_cluster_f64(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" :: "r"(addr), "d"(v) : "memory");
}

__global__ void __launch_bounds__(kSumThreads)
    stats_summary_kernel(int64_t rows, const float* __restrict__ st, const uint8_t* __restrict__ mask,
                         const int32_t* __restrict__ token_traj, int32_t n_traj, const float* __restrict__ coef,
                         double* __restrict__ out, double* slots, uint32_t* done, int32_t* status) {
  __shared__ double part[kSumThreads / 32][5];
  __shared__ double cta_total[kSumCluster][5];  // used in rank 0
  const uint32_t rank = cluster_ctarank();
  const unsigned C = cluster_nctarank(), cid = blockIdx.x / C, ncl = gridDim.x / C;
  const int64_t G = static_cast<int64_t>(gridDim.x) * kSumThreads;
  double acc[3] = {0.0, 0.0, 0.0};  // H, KL, rho
  double clip = 0.0;                // flags other than 0 and 1
  unsigned n_rows = 0, n_clip = 0;  // at most rows / G each
  bool bad = false;
  auto add_rows = [&](int64_t r0, int nr) {  // rows r0, r0 + G, ... (nr <= kSumUnroll of them)
    uint32_t m[kSumUnroll];
    int32_t i[kSumUnroll];
#pragma unroll
    for (int k = 0; k < kSumUnroll; ++k) {
      m[k] = k < nr ? mask[r0 + k * G] : 0u;
      i[k] = k < nr ? token_traj[r0 + k * G] : 0;
    }
    float c[kSumUnroll];
#pragma unroll
    for (int k = 0; k < kSumUnroll; ++k) {
      const bool in = i[k] >= 0 && i[k] < n_traj;
      bad |= m[k] != 0 && !in;
      c[k] = (m[k] != 0 && in) ? coef[i[k]] : 0.f;
    }
    float v[kSumUnroll][4];
#pragma unroll
    for (int k = 0; k < kSumUnroll; ++k) {
      const float* s = st + (r0 + k * G) * 5;
#pragma unroll
      for (int q = 0; q < 4; ++q) v[k][q] = c[k] != 0.f ? s[q + 1] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kSumUnroll; ++k) {
      if (c[k] == 0.f) continue;
      ++n_rows;
      if (v[k][1] == 1.f) ++n_clip;
      else if (v[k][1] != 0.f) clip += static_cast<double>(v[k][1]);
      acc[0] += widen(v[k][2]);  // H
      acc[1] += widen(v[k][3]);  // KL
      acc[2] += widen(v[k][0]);  // rho
    }
  };
  int64_t r = static_cast<int64_t>(blockIdx.x) * kSumThreads + threadIdx.x;
  for (; r + (kSumUnroll - 1) * G < rows; r += kSumUnroll * G) add_rows(r, kSumUnroll);
  if (r < rows) add_rows(r, static_cast<int>((rows - r + G - 1) / G));
  if (bad) flag_status(status, RL_DEV_BAD_TRAJ);
  const unsigned wr = __reduce_add_sync(0xffffffffu, n_rows), wc = __reduce_add_sync(0xffffffffu, n_clip);
#pragma unroll
  for (int k = 0; k < 3; ++k) acc[k] = warp_sum(acc[k]);
  if (__any_sync(0xffffffffu, clip != 0.0)) clip = warp_sum(clip);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) {
    part[warp][0] = static_cast<double>(wr);
    part[warp][1] = static_cast<double>(wc) + clip;
    part[warp][2] = acc[0];
    part[warp][3] = acc[1];
    part[warp][4] = acc[2];
  }
  cluster_sync_all();  // every CTA of the cluster is running before rank 0's memory is written
  if (threadIdx.x < 5) {
    double sum = 0.0;
    for (int w = 0; w < kSumThreads / 32; ++w) sum += part[w][threadIdx.x];
    st_cluster_f64(map_to_rank(smem_addr(&cta_total[rank][threadIdx.x]), 0), sum);
  }
  cluster_sync_all();
  if (rank != 0 || warp != 0) return;
  if (lane < 5) {
    double sum = 0.0;
    for (unsigned k = 0; k < C; ++k) sum += cta_total[k][lane];
    if (ncl == 1) {
      out[lane] += sum;
      return;
    }
    slots[cid * 5 + lane] = sum;
    __threadfence();
  }
  if (ncl == 1) return;
  __syncwarp();
  unsigned last = 0;
  if (lane == 0) last = atomicAdd(done, 1u) == ncl - 1 ? 1u : 0u;
  last = __shfl_sync(0xffffffffu, last, 0);
  if (!last) return;
  __threadfence();
  if (lane < 5) {
    double sum = 0.0;
    for (unsigned k = 0; k < ncl; ++k) sum += __ldcg(slots + k * 5 + lane);
    out[lane] += sum;
  }
  if (lane == 0) *done = 0u;
}

}  // namespace rl

extern "C" rl_status rl_token_stats_summary(int64_t rows, const float* token_stats, const uint8_t* mask,
                                            const int32_t* token_traj, int32_t n_traj, const float* coef,
                                            double* summary_accum, void* ws, size_t ws_bytes, rl_stream_t stream) {
  using namespace rl;
  clear_error();
  if (rows < 0 || n_traj < 0) return set_error(RL_ERR_INVALID_ARG, "rl_token_stats_summary: negative size");
  if (!summary_accum || !ws) return set_error(RL_ERR_INVALID_ARG, "rl_token_stats_summary: NULL argument");
  if (ws_bytes < kWsHeader) return set_error(RL_ERR_WORKSPACE_TOO_SMALL, "rl_token_stats_summary: workspace too small");
  if (rows == 0) return RL_OK;
  if (!token_stats || !mask || !token_traj || (n_traj > 0 && !coef))
    return set_error(RL_ERR_INVALID_ARG, "rl_token_stats_summary: NULL array argument");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  auto kern = stats_summary_kernel;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kSumCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(kSumCluster);
  cfg.blockDim = dim3(kSumThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static std::mutex mu;
  static std::map<int, unsigned> width;  // by device: CTAs of a cluster
  unsigned C = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = width.find(dev);
    if (it == width.end()) {
      // clusters of 16 are not portable: a partition of a GPU may have no 16 SMs in one GPC
      int fit = 0;
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&fit, kern, &cfg);
      if (e != cudaSuccess) {
        (void)cudaGetLastError();
        fit = 0;
      }
      it = width.emplace(dev, fit > 0 ? kSumCluster : kSumCluster / 2).first;
    }
    C = it->second;
  }
  // a cluster per 8,192 rows up to the five that have a slot: below that a second cluster's
  // trip through the slots costs more than the rows it takes over
  // (a workspace whose slots are not on 8-byte boundaries has one cluster, which needs none)
  const int64_t clusters =
      reinterpret_cast<uintptr_t>(ws) % 8 != 0 ? 1 : std::min<int64_t>(kSumSlots, (rows + 8191) / 8192);
  attr[0].val.clusterDim.x = C;
  cfg.gridDim = dim3(static_cast<unsigned>(clusters) * C);
  char* wsb = static_cast<char*>(ws);
  e = cudaLaunchKernelEx(&cfg, kern, rows, token_stats, mask, token_traj, n_traj, coef, summary_accum,
                         reinterpret_cast<double*>(wsb + kWsSummaryOffset),
                         reinterpret_cast<uint32_t*>(wsb + kWsSummaryDoneOffset), reinterpret_cast<int32_t*>(ws));
  if (e != cudaSuccess) return cuda_error(e, "stats_summary_kernel launch");
  return RL_OK;
}
