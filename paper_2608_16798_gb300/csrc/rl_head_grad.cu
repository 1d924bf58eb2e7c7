// Backward products of the fused LM head on the tensor cores (tcgen05, CTA pairs), both in
// one persistent launch:
//
//   dH  = dZ W      M = tokens, N = D, K = V        A = dZ   (K-major: V contiguous)
//                                                   B = W    (MN-major: D contiguous)
//   dW += dZ^T H    M = V,      N = D, K = tokens   A = dZ^T (MN-major: V contiguous)
//                                                   B = H    (MN-major: D contiguous)
//
// dZ is the bf16 gradient of the logits of a chunk (or group of chunks) of n tokens, formed
// in the workspace by the loss pass; W and H are the caller's bf16 matrices in their own
// row-major layouts, read in place (the MN-major operands use the transpose bits of the
// instruction descriptor: nothing is transposed in memory).
//
// A 2-CTA cluster computes output tiles of 256 rows x 512 columns: per K step of 16 the even
// CTA issues two cta_group::2 MMAs of 256 x 256 that share the A operand, into one fp32
// accumulator of all 512 TMEM columns (each CTA holds 128 rows of A and, for each MMA, 128 of
// B's 256 columns; 4 shared-memory stages of 48 KB filled by TMA; both CTAs' loads complete on
// the even CTA's barrier and the MMA's commits are multicast to both). Sharing A between two
// MMAs moves a quarter fewer operand bytes through shared memory and L2 per flop than 256 x
// 256 tiles, which is what lets the MMAs run close to their peak rate. The epilogue drains
// TMEM 32 columns at a time: a dW tile into a swizzled shared-memory slab, which the TMA adds to the
// fp32 d_weight (a tiled reduce-add); a dH tile from the registers to its tokens' rows of d_hidden (bf16
// or fp32), or to a part's sums.
//
// Work items are dH tiles (each the whole contraction over V: long) followed by dW tiles
// (contraction over the n tokens: short), handed out by a counter in global memory as pairs
// become free: the dW tiles fill the time the last dH tiles leave over, and pairs that run at
// the same time work on neighbouring tiles, sharing operand rows and columns in L2. The even
// CTA's producer thread takes each item and publishes it to both CTAs' roles through a small
// ring guarded by mbarriers. Every output element receives exactly one store (dH) or one
// addition (dW) per launch, so results do not depend on the schedule.
#include <cuda.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "rl_device.cuh"
#include "rl_head_tokens.cuh"
#include "rl_host.h"
#include "rl_tc.cuh"
#include "rl_tmap.h"

namespace rl {
namespace grad {

constexpr int BM = 128;                          // output rows per CTA (TMEM lanes)
constexpr int NB = 512;                          // output columns per tile (TMEM columns)
constexpr int NH = NB / 256;                     // MMAs per K step (N = 256 each)
constexpr int BK = 64;                           // contraction elements per stage
constexpr uint32_t A_BYTES = BM * BK * 2;        // this CTA's 128 rows of A
constexpr uint32_t HALF_BYTES = 64 * BK * 2;     // one 64-element MN block of 64 K rows
constexpr uint32_t B_BYTES = NH * 2 * HALF_BYTES;  // this CTA's 128 columns of each MMA's B
constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int NS = 4;                            // shared-memory stages
constexpr int NR = 4;                            // slots of the work-item ring
constexpr uint32_t SLAB_BYTES = 4096;            // epilogue slab: 32 rows x 128 bytes
constexpr int kThreads = 192;                    // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue
constexpr size_t kSmem = NS * STAGE_BYTES + 4 * 2 * SLAB_BYTES + 1024;
static_assert(kSmem <= 232448 - 1024, "shared memory of the backward kernel");
// consumers of each published work item: the MMA thread and 4 epilogue warps of the even CTA,
// the producer thread and 4 epilogue warps of the odd CTA
constexpr uint32_t kItemReaders = 10;

struct GradArgs {
  Tokens tok;
  int32_t group;         // which group of tokens
  int32_t D;
  int32_t n_w;           // dW tiles: row tiles x n_nt
  int32_t n_nt;          // 512-column tiles of D
  int32_t nkb_h;         // 64-element K blocks over V (dH)
  int32_t parts;         // parts of that contraction, each an item
  float* part_sums;      // [parts][Tc x D] with parts > 1 (one chunk per group then)
  void* d_hidden;        // [T x D]
  uint32_t* counter;     // work-item counter (zero at launch)
  const double* row_loss;  // [T] loss contributions
  double* loss_accum;    // the caller's total in the call's last launch, else null
  int32_t* status;
};

// Element type of the stored d_hidden tiles.
enum HOut { H_F32 = 0, H_BF16 = 1 };

// The tokens' loss contributions added in a fixed order into the caller's total by the four epilogue
// warps of CTA 0, while its first accumulator fills (at 500 tokens a launch of its own took 8 us, the
// rescale's last CTA 5).
// Thread k adds tokens k, k + 128, ... into eight accumulators in turn (eight loads in flight).
__device__ __forceinline__ void sum_loss(const GradArgs& p) {
  __shared__ double part[4];
  const int k = static_cast<int>(threadIdx.x) - 64;
  double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int64_t t = k;
  for (; t + 7 * 128 < p.tok.T; t += 8 * 128) {
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i] += p.row_loss[t + i * 128];
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (t + i * 128 < p.tok.T) acc[i] += p.row_loss[t + i * 128];
  const double s = warp_sum(((acc[0] + acc[1]) + (acc[2] + acc[3])) + ((acc[4] + acc[5]) + (acc[6] + acc[7])));
  if ((k & 31) == 0) part[k >> 5] = s;
  asm volatile("bar.sync 1, 128;" ::: "memory");
  if (k == 0) *p.loss_accum += (part[0] + part[1]) + (part[2] + part[3]);
}

template <int HO>
__global__ void __launch_bounds__(kThreads, 1) head_grad_kernel(
    const __grid_constant__ CUtensorMap tmAh, const __grid_constant__ CUtensorMap tmBh,
    const __grid_constant__ CUtensorMap tmAw, const __grid_constant__ CUtensorMap tmBw,
    const __grid_constant__ CUtensorMap tmOw, const GradArgs p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[NS], empty[NS], accf, acce, ifull[NR], iempty[NR];
  __shared__ int32_t ring[NR];
  __shared__ uint32_t tbase;
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* slabs = sm + NS * STAGE_BYTES;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  // the group's tokens, its dH tiles (row tiles x n_nt) and the dW tiles' K blocks
  const Chunk grp = group_of(p.tok, p.group);
  const bool sums_loss = p.loss_accum != nullptr && blockIdx.x == 0 && warp >= 2;
  if (grp.count == 0) {  // the whole grid: nothing to multiply
    if (sums_loss) sum_loss(p);
    return;
  }
  const int n_h1 = (grp.count + 2 * BM - 1) / (2 * BM) * p.n_nt;
  const int n_h = n_h1 * p.parts;
  const int nkb_w = (grp.count + BK - 1) / BK;
  const int n_items = n_h + p.n_w;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accf, 1);
    mbar_init(&acce, 8);  // 4 epilogue warps in each CTA of the pair
    for (int r = 0; r < NR; ++r) {
      mbar_init(&ifull[r], 1);
      mbar_init(&iempty[r], kItemReaders);
    }
    fence_mbar_init();
  }
  if (warp == 1) tc::tmem_alloc_pair(&tbase, NB);
  tc::fence_before_sync();
  cluster_sync_all();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;

  // item -> (dW?, tile row, tile column, first K block, K blocks); columns fastest, then rows, then
  // the parts of dH's contraction
  const int n_nt = p.n_nt, nkb_h = p.nkb_h, parts = p.parts;
  auto decode = [=](int item, bool& w, int& mt, int& nt, int& kb0, int& nkb) {
    w = item >= n_h;
    const int part = w ? 0 : item / n_h1;
    const int r = w ? item - n_h : item % n_h1;
    mt = r / n_nt;
    nt = r % n_nt;
    kb0 = static_cast<int>(static_cast<int64_t>(part) * nkb_h / parts);
    nkb = w ? nkb_w : static_cast<int>(static_cast<int64_t>(part + 1) * nkb_h / parts) - kb0;
  };
  // Read the k-th published item (every role but the even CTA's producer): -1 if the wait
  // ran out.
  auto next_item = [&](uint32_t k) -> int {
    const int r = static_cast<int>(k % NR);
    const bool got = rank == 0 ? mbar_wait_bounded(&ifull[r], (k / NR) & 1)
                               : mbar_wait_cluster_bounded(&ifull[r], (k / NR) & 1);
    if (!got) return -1;
    const int item = ring[r];
    if (rank == 0) mbar_arrive(&iempty[r]);
    else mbar_arrive_remote(map_to_rank(smem_addr(&iempty[r]), 0));
    return item;
  };

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      for (uint32_t k = 0; ok; ++k) {
        int item;
        if (rank == 0) {
          // take the next item and publish it to both CTAs
          const int r = static_cast<int>(k % NR);
          if (k >= NR && !mbar_wait_cluster_bounded(&iempty[r], ((k / NR) - 1) & 1)) {
            flag_status(p.status, RL_DEV_TIMEOUT);
            break;
          }
          const uint32_t v = atomicAdd(p.counter, 1u);
          item = v < static_cast<uint32_t>(n_items) ? static_cast<int>(v) : n_items;
          ring[r] = item;
          const uint32_t peer_slot = map_to_rank(smem_addr(&ring[r]), 1);
          asm volatile("st.shared::cluster.u32 [%0], %1;" :: "r"(peer_slot), "r"(item) : "memory");
          mbar_arrive(&ifull[r]);
          mbar_arrive_remote(map_to_rank(smem_addr(&ifull[r]), 1));
        } else {
          item = next_item(k);
          if (item < 0) {
            flag_status(p.status, RL_DEV_TIMEOUT);
            break;
          }
        }
        if (item >= n_items) break;
        bool w;
        int mt, nt, kb0, nkb;
        decode(item, w, mt, nt, kb0, nkb);
        const int m0 = mt * 2 * BM + static_cast<int>(rank) * BM;
        const int n0 = nt * NB + static_cast<int>(rank) * 128;
        const CUtensorMap* mb = w ? &tmBw : &tmBh;
        for (int kb = 0; kb < nkb; ++kb, ++g) {
          const int s = g % NS;
          const int k0 = (kb0 + kb) * BK;
          const uint32_t use = g / NS;
          if (use > 0 && !mbar_wait_bounded(&empty[s], (use - 1) & 1)) {
            flag_status(p.status, RL_DEV_TIMEOUT);
            ok = false;
            break;
          }
          uint8_t* st = sm + s * STAGE_BYTES;
          if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * STAGE_BYTES);  // both CTAs' bytes
          const uint32_t bar = map_to_rank(smem_addr(&full[s]), 0);
          if (w) {
            tc::tma_load_2d_pair(st, &tmAw, m0, k0, bar);
            tc::tma_load_2d_pair(st + HALF_BYTES, &tmAw, m0 + 64, k0, bar);
          } else {
            tc::tma_load_2d_pair(st, &tmAh, k0, m0, bar);
          }
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            uint8_t* sb = st + A_BYTES + h * 2 * HALF_BYTES;
            tc::tma_load_2d_pair(sb, mb, n0 + h * 256, k0, bar);
            tc::tma_load_2d_pair(sb + HALF_BYTES, mb, n0 + h * 256 + 64, k0, bar);
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc_h = tc::idesc_bf16_f32_major(2 * BM, 256, false, true);
      constexpr uint32_t idesc_w = tc::idesc_bf16_f32_major(2 * BM, 256, true, true);
      uint32_t g = 0;
      for (uint32_t t = 0;; ++t) {
        const int item = next_item(t);
        if (item < 0) {
          flag_status(p.status, RL_DEV_TIMEOUT);
          break;
        }
        if (item >= n_items) break;
        bool w;
        int mt, nt, kb0, nkb;
        decode(item, w, mt, nt, kb0, nkb);
        if (t > 0 && !mbar_wait_cluster_bounded(&acce, (t - 1) & 1)) {
          flag_status(p.status, RL_DEV_TIMEOUT);
          break;
        }
        tc::fence_after_sync();
        const uint32_t idesc = w ? idesc_w : idesc_h;
        bool ok = true;
        for (int kb = 0; kb < nkb; ++kb, ++g) {
          const int s = g % NS;
          if (!mbar_wait_bounded(&full[s], (g / NS) & 1)) {
            flag_status(p.status, RL_DEV_TIMEOUT);
            ok = false;
            break;
          }
          tc::fence_after_sync();
          const uint32_t a = smem_addr(sm + s * STAGE_BYTES), b = a + A_BYTES;
#pragma unroll
          for (int k = 0; k < BK / 16; ++k) {
            const uint64_t ad = w ? tc::desc_mnmajor_sw128(a + k * 2048, HALF_BYTES, 1024)
                                  : tc::desc_kmajor_sw128(a + k * 32);
#pragma unroll
            for (int h = 0; h < NH; ++h) {
              const uint64_t bd = tc::desc_mnmajor_sw128(b + h * 2 * HALF_BYTES + k * 2048, HALF_BYTES, 1024);
              tc::mma_bf16_pair(tmem + h * 256, ad, bd, idesc, (kb | k) != 0 ? 1u : 0u);
            }
          }
          tc::mma_commit_pair(&empty[s], 0x3);
        }
        if (!ok) break;
        tc::mma_commit_pair(&accf, 0x3);
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue (4 warps)
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    uint8_t* my = slabs + (warp - 2) * 2 * SLAB_BYTES;
    const uint32_t tq = tmem + (static_cast<uint32_t>(32 * q) << 16);
    uint32_t buf = 0;
    if (sums_loss) sum_loss(p);
    for (uint32_t t = 0;; ++t) {
      int item = 0;
      if (lane == 0) item = next_item(t);
      item = __shfl_sync(0xffffffffu, item, 0);
      if (item < 0) {
        if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
        break;
      }
      if (item >= n_items) break;
      bool w;
      int mt, nt, kb0, nkb;
      decode(item, w, mt, nt, kb0, nkb);
      if (!mbar_wait_sleep_bounded(&accf, t & 1)) {
        if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
        break;
      }
      tc::fence_after_sync();
      const int row0 = mt * 2 * BM + static_cast<int>(rank) * BM + 32 * q;
      // dH: lane l holds row row0 + l, which goes straight to its token's row of d_hidden, or, as
      // one of several parts, to its row of the part's sums
      const int hr = row0 + lane;
      const bool h_ok = !w && hr < grp.count;
      const bool in_parts = parts > 1;
      int64_t h_at = 0;
      if (h_ok)
        h_at = (in_parts ? static_cast<int64_t>(item / n_h1) * p.tok.Tc + hr
                         : static_cast<int64_t>(token_of(p.tok, grp, hr))) * p.D + nt * NB;
#pragma unroll 1
      for (int c = 0; c < NB / 32; ++c) {
        float v[32];
        tc::tmem_ld32(tq + c * 32, v);
        if (c == NB / 32 - 1) {
          // the whole accumulator is in registers or slabs: hand it back to the MMA
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) {
            if (rank != 0) mbar_arrive_remote(map_to_rank(smem_addr(&acce), 0));
            else mbar_arrive(&acce);
          }
        }
        if (!w) {
          if (h_ok && nt * NB + c * 32 < p.D) {  // neither past the tokens nor past D's last tile
            if (HO == H_BF16 && !in_parts) {
              uint16_t* out = static_cast<uint16_t*>(p.d_hidden) + h_at + c * 32;
#pragma unroll
              for (int j = 0; j < 4; ++j)
                *reinterpret_cast<uint4*>(out + 8 * j) =
                    make_uint4(pack_bf16x2(v[8 * j], v[8 * j + 1]), pack_bf16x2(v[8 * j + 2], v[8 * j + 3]),
                               pack_bf16x2(v[8 * j + 4], v[8 * j + 5]), pack_bf16x2(v[8 * j + 6], v[8 * j + 7]));
            } else {
              float* out = (in_parts ? p.part_sums : static_cast<float*>(p.d_hidden)) + h_at + c * 32;
#pragma unroll
              for (int j = 0; j < 8; ++j)
                *reinterpret_cast<float4*>(out + 4 * j) =
                    make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
            }
          }
          __syncwarp();  // the next TMEM load is the whole warp's
          continue;
        }
        uint8_t* sb = my + buf * SLAB_BYTES;
        if (lane == 0) tc::bulk_wait_read_1();  // the slab's previous TMA has read it
        __syncwarp();
        // 32 rows x 128 bytes, 128-byte swizzle: 16-byte chunk j of row r at chunk j ^ (r % 8)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<float4*>(sb + lane * 128 + ((j ^ (lane & 7)) << 4)) =
              make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tc::tma_reduce_add_2d(&tmOw, nt * NB + c * 32, row0, sb);
          bulk_commit();
        }
        buf ^= 1;
      }
    }
    if (lane == 0) tc::bulk_wait_all();
  }
  tc::fence_before_sync();
  cluster_sync_all();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc_pair(tmem, NB);
  }
}

// dH from its parts: the fp32 sums of the parts of the contraction over V added in order, into the
// token's row of d_hidden. Grid-stride over rows, four columns per thread and step.
template <int HO>
__global__ void __launch_bounds__(256) head_combine_kernel(const GradArgs p) {
  const Chunk grp = group_of(p.tok, p.group);
  const int64_t per_part = static_cast<int64_t>(p.tok.Tc) * p.D;
  for (int r = blockIdx.x; r < grp.count; r += gridDim.x) {
    const int64_t to = static_cast<int64_t>(token_of(p.tok, grp, r)) * p.D;
    for (int c = threadIdx.x * 4; c < p.D; c += 1024) {
      const float* src = p.part_sums + static_cast<int64_t>(r) * p.D + c;
      float4 a = *reinterpret_cast<const float4*>(src);
#pragma unroll 4
      for (int k = 1; k < p.parts; ++k) {
        const float4 b = *reinterpret_cast<const float4*>(src + k * per_part);
        a.x += b.x;
        a.y += b.y;
        a.z += b.z;
        a.w += b.w;
      }
      if (HO == H_BF16)
        *reinterpret_cast<uint2*>(static_cast<uint16_t*>(p.d_hidden) + to + c) =
            make_uint2(pack_bf16x2(a.x, a.y), pack_bf16x2(a.z, a.w));
      else
        *reinterpret_cast<float4*>(static_cast<float*>(p.d_hidden) + to + c) = a;
    }
  }
}

}  // namespace grad

rl_status head_grad(const Tokens& tok, int group, int64_t rows, const uint16_t* dz, int64_t ldz, int64_t V,
                    const void* weight, const void* hidden, int64_t D, void* d_hidden, rl_dtype dh_dtype,
                    float* d_weight, float* part_sums, int parts, const double* row_loss, double* loss_accum,
                    uint32_t* counter, int32_t* status, cudaStream_t s) {
  using namespace grad;
  CUtensorMap ah, bh, aw, bw, ow;
  const bool bf16 = dh_dtype == RL_BF16;
  rl_status st =
      tmap_2d(&ah, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, dz, V, rows, ldz * 2, BK, BM, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == RL_OK)
    st = tmap_2d(&bh, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, weight, D, V, D * 2, 64, BK, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == RL_OK)
    st = tmap_2d(&aw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, dz, V, rows, ldz * 2, 64, BK, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == RL_OK)
    st = tmap_2d(&bw, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, hidden, D, rows, D * 2, 64, BK, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st == RL_OK)
    st = tmap_2d(&ow, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, d_weight, D, V, D * 4, 32, 32, CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != RL_OK) return st;
  GradArgs a = {};
  a.tok = tok;
  a.group = group;
  a.D = static_cast<int32_t>(D);
  a.n_nt = static_cast<int32_t>((D + NB - 1) / NB);
  a.n_w = static_cast<int32_t>((V + 2 * BM - 1) / (2 * BM)) * a.n_nt;
  a.nkb_h = static_cast<int32_t>((V + BK - 1) / BK);
  a.parts = parts;
  a.part_sums = part_sums;
  a.d_hidden = d_hidden;
  a.counter = counter;
  a.row_loss = row_loss;
  a.loss_accum = loss_accum;
  a.status = status;
  const int32_t n_h = static_cast<int32_t>((rows + 2 * BM - 1) / (2 * BM)) * a.n_nt * parts;  // at most

  auto kern = bf16 ? head_grad_kernel<H_BF16> : head_grad_kernel<H_F32>;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaGetDevice");
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static std::mutex mu;
  static std::map<std::pair<int, bool>, int> resident;  // CTA pairs resident at once
  int max_pairs = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    const auto key = std::make_pair(dev, bf16);
    auto it = resident.find(key);
    if (it == resident.end()) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmem));
      if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(head_grad_kernel)");
      int npairs = 0;
      cfg.gridDim = dim3(2);
      e = cudaOccupancyMaxActiveClusters(&npairs, kern, &cfg);
      if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveClusters(head_grad_kernel)");
      if (npairs <= 0) return set_error(RL_ERR_UNSUPPORTED, "head_grad_kernel: no CTA pair fits on the device");
      it = resident.emplace(key, npairs).first;
    }
    max_pairs = it->second;
  }
  // persistent: at most as many pairs as fit on the device at once, and no more than items
  cfg.gridDim = dim3(2 * std::max(1, std::min(n_h + a.n_w, max_pairs)));
  e = cudaLaunchKernelEx(&cfg, kern, ah, bh, aw, bw, ow, a);
  if (e != cudaSuccess) return cuda_error(e, "cudaLaunchKernelEx(head_grad_kernel)");
  if (parts > 1) {
    auto combine = bf16 ? head_combine_kernel<H_BF16> : head_combine_kernel<H_F32>;
    combine<<<static_cast<unsigned>(std::min<int64_t>(rows, 152 * 8)), 256, 0, s>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "head_combine_kernel launch");
  }
  return RL_OK;
}

}  // namespace rl
