// Fused LM head: the policy loss and its gradients with respect to the hidden states
// and the output projection, with the logits Z = H W^T never written to memory.
//
// Only the tokens that are trained on go through the products: head_select_kernel lists them, and
// for each chunk of the list:
//   0. head_gather_kernel   packs the chunk's hidden states.
//   1. head_kernel<STATS_P> tcgen05 GEMM tiles Z[256 x 256] = H W^T on CTA pairs (2-CTA
//      clusters, cta_group::2 MMAs; TMA-fed shared-memory stages, fp32 accumulators in TMEM,
//      two accumulators so the epilogue of one tile overlaps the MMAs of the next; each CTA
//      holds 128 of the tile's tokens). The epilogue reads each tile twice from TMEM: first
//      its row maximum m_j, then e = exp(z - m_j), which it stores (bf16) in the chunk's
//      dZ buffer, with m_j per token and tile, and folds into per-row online-softmax
//      partials: two per block of 4,096 entries (its even and its odd tiles).
//   2. head_dz_kernel       merges each token's partials into lse, entropy and logp (one warp),
//      evaluates the objective's per-token terms (same readings as the logits path), writes the
//      token's loss contribution, and rescales the stored e in place into
//      dZ = c [g (delta_a - p) + alpha p (log p + H)], p = e exp(m_j - lse) (HBM-bound: the
//      logits are formed once, not twice).
// The dZ of one chunk (4,096 tokens x V in bf16) is the only logits-sized buffer; a caller
// that passes more workspace lets a group of several chunks keep their dZ side by side.
// After the group's last chunk (every chunk, with the smallest workspace):
//   3. dH = dZ W and dW += dZ^T H over the group in one persistent launch of
//      head_grad_kernel (rl_head_grad.cu): CTA-pair tcgen05 MMAs on 256 x 512 tiles with the
//      operands in their row-major layouts (dZ K-major for dH, MN-major for dW; W and H
//      MN-major), dH tiles first and dW tiles after them, handed out by a work counter; dH rows
//      are stored at their tokens' places (a short call's in parts of the contraction, which
//      head_combine_kernel adds), dW added in fp32 by TMA reduce-add, once per group. The last
//      group's launch also sums the loss.
// The forward-only call runs head_wide_kernel<STATS> (256 x 512 tiles, no stores; the same
// partials) and head_logp_merge_kernel.
// A token's statistics are summed in one order whatever the call's size and workspace: tiles j, j + 2,
// ... of a block of 16 in turn, then the blocks' partials. Short calls, whose work items are smaller
// than a block, leave every tile's own partial and the merge takes the first step too.
// The objective (Sec. 2.3.2, Sec. 3.2.4) is the same as for rl_policy_loss_fwd_bwd; here
// pi_theta's logits come from the hidden states times the vocabulary projection.
#include <cuda.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>

#include "rl_device.cuh"
#include "rl_head_tokens.cuh"
#include "rl_host.h"
#include "rl_tc.cuh"
#include "rl_tmap.h"

namespace rl {
namespace head {

constexpr int BM = 128;            // tokens per tile (TMEM lanes)
constexpr int BN = 256;            // vocabulary entries per tile (TMEM columns per accumulator)
constexpr int BK = 64;             // hidden elements per stage (one 128-byte swizzle row)
constexpr int NS = 4;              // shared-memory stages
constexpr int kMaxVb = 16;         // most N tiles per work item (16: a vocabulary block of 4,096)
constexpr int kPairs = 76;         // CTA pairs of the GPU (152 SMs)
constexpr uint32_t A_BYTES = BM * BK * 2, B_BYTES = BN * BK * 2, STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int kThreads = 192;      // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue
constexpr size_t kSmem = NS * STAGE_BYTES + 1024;
// CTA-pair form: each CTA stages its 128 tokens and half of the 256 vocabulary rows
#ifndef RL_HEAD_NS2
#define RL_HEAD_NS2 6
#endif
constexpr int NS2 = RL_HEAD_NS2;
constexpr uint32_t STAGE2_BYTES = A_BYTES + B_BYTES / 2;
constexpr size_t kSmem2 = NS2 * STAGE2_BYTES + 1024;
#ifndef RL_HEAD_PAIR
#define RL_HEAD_PAIR 1
#endif
constexpr bool kPair = RL_HEAD_PAIR != 0;
constexpr uint32_t kWBoxRows = kPair ? BN / 2 : BN;  // rows of W per TMA box
#ifndef RL_HEAD_CHUNK
#define RL_HEAD_CHUNK 4096
#endif
constexpr int64_t kChunk = RL_HEAD_CHUNK;  // tokens per chunk (tuning knob, compile time)
constexpr int64_t kParts = 2;               // partials per token and block of 16 tiles (even, odd ones)

enum Mode { STATS = 0, STATS_P = 1 };

// Per-token coefficients of dZ (formed by head_dz_kernel).
struct RowCoef {
  float nlse2;  // -lse * log2(e)
  float Kp;     // dZ_v = Kp p_v (+ cg at v = a), without the entropy term
  float cg;
  float ca;     // entropy: dZ_v = p_v (ca z_v + Ke) (+ cg at v = a)
  float Ke;
  int32_t a;
  int32_t active;
};

struct HeadArgs {
  Tokens tok;  // the call's tokens
  int32_t chunk;           // which chunk of them
  int32_t D, V, vb_tiles, n_vb, n_nt;  // N tiles per work item (even), items and tiles per row tile
  int32_t ent;
  const int32_t* token_ids;
  float4* partials;        // (m, s, u, z_a): [2 n_vb][Tc], a block's even tiles, then its odd ones, or [n_nt][Tc]
  uint16_t* dz;            // [G Tc x ldz] bf16: e = exp(z - m_j) (STATS_P), the group's chunks in turn
  int64_t ldz;
  float* tmax;             // [Tc x n_nt]: m_j per token and tile (STATS_P)
  int32_t* status;
};

// Two forms share this kernel. PAIR = false: each CTA computes 128 x 256 tiles with
// cta_group::1 MMAs from 48 KB stages (A 16 KB + B 32 KB, 4 stages). PAIR = true: a cluster of
// two CTAs computes 256 x 256 tiles with cta_group::2 MMAs issued by the even CTA; each CTA
// loads its own 128 tokens of H and its own 128 vocabulary rows of W (32 KB stages, 6 of them),
// both CTAs' loads complete on the even CTA's barrier, the MMA's commits are multicast to both
// CTAs, and each CTA's epilogue drains its own 128 TMEM lanes (all 256 columns) and tells the
// even CTA's MMA thread when an accumulator is free. Per pair this halves the W operand each SM
// fetches and stages per MMA.
template <int MODE, bool PAIR, bool TILE_PARTS>
__global__ void __launch_bounds__(kThreads, 1) head_kernel(const __grid_constant__ CUtensorMap tmH,
                                                           const __grid_constant__ CUtensorMap tmW,
                                                           const HeadArgs p) {
  constexpr int kNS = PAIR ? NS2 : NS;
  constexpr uint32_t kStage = PAIR ? STAGE2_BYTES : STAGE_BYTES;
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[kNS], empty[kNS], accf[2], acce[2];
  __shared__ uint32_t tbase;
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  const int unit = PAIR ? static_cast<int>(blockIdx.x >> 1) : static_cast<int>(blockIdx.x);
  const int n_units = PAIR ? static_cast<int>(gridDim.x >> 1) : static_cast<int>(gridDim.x);
  constexpr int kMStep = PAIR ? 2 * BM : BM;  // tokens per work item
  const Chunk ch = chunk_of(p.tok, p.chunk);
  const int n_m = (ch.count + kMStep - 1) / kMStep;
  const int n_items = n_m * p.n_vb;
  const int nkb = p.D / BK;
  if (n_items == 0) return;  // the whole grid: no token of this chunk is trained on

  if (threadIdx.x == 0) {
    for (int s = 0; s < kNS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], PAIR ? 8 : 4);
    }
    fence_mbar_init();
  }
  if (warp == 1) {
    if constexpr (PAIR) tc::tmem_alloc_pair(&tbase, 2 * BN);
    else tc::tmem_alloc(&tbase, 2 * BN);
  }
  tc::fence_before_sync();
  if constexpr (PAIR) cluster_sync_all();
  else __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      for (int item = unit; item < n_items && ok; item += n_units) {
        const int vb = item / n_m, m0 = (item % n_m) * kMStep + static_cast<int>(rank) * BM;
        const int nt1 = min((vb + 1) * p.vb_tiles, p.n_nt);
        for (int nt = vb * p.vb_tiles; nt < nt1 && ok; ++nt) {
          for (int kb = 0; kb < nkb; ++kb, ++g) {
            const int s = g % kNS;
            const uint32_t use = g / kNS;
            if (use > 0 && !mbar_wait_bounded(&empty[s], (use - 1) & 1)) {
              flag_status(p.status, RL_DEV_TIMEOUT);
              ok = false;
              break;
            }
            uint8_t* st = sm + s * kStage;
            if constexpr (PAIR) {
              if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * kStage);  // both CTAs' bytes
              const uint32_t bar = map_to_rank(smem_addr(&full[s]), 0);
              tc::tma_load_2d_pair(st, &tmH, kb * BK, ch.row + m0, bar);
              tc::tma_load_2d_pair(st + A_BYTES, &tmW, kb * BK, nt * BN + static_cast<int>(rank) * (BN / 2), bar);
            } else {
              mbar_arrive_expect_tx(&full[s], kStage);
              tc::tma_load_2d(st, &tmH, kb * BK, ch.row + m0, &full[s]);
              tc::tma_load_2d(st + A_BYTES, &tmW, kb * BK, nt * BN, &full[s]);
            }
          }
        }
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16_f32(kMStep, BN);
      uint32_t g = 0, t = 0;
      bool ok = true;
      for (int item = unit; item < n_items && ok; item += n_units) {
        const int vb = item / n_m;
        const int nt1 = min((vb + 1) * p.vb_tiles, p.n_nt);
        for (int nt = vb * p.vb_tiles; nt < nt1 && ok; ++nt, ++t) {
          const int acc = t & 1;
          if (t >= 2) {
            const uint32_t par = ((t >> 1) - 1) & 1;
            const bool got = PAIR ? mbar_wait_cluster_bounded(&acce[acc], par) : mbar_wait_bounded(&acce[acc], par);
            if (!got) {
              flag_status(p.status, RL_DEV_TIMEOUT);
              ok = false;
              break;
            }
          }
          tc::fence_after_sync();
          const uint32_t d = tmem + acc * BN;
          for (int kb = 0; kb < nkb; ++kb, ++g) {
            const int s = g % kNS;
            if (!mbar_wait_bounded(&full[s], (g / kNS) & 1)) {
              flag_status(p.status, RL_DEV_TIMEOUT);
              ok = false;
              break;
            }
            tc::fence_after_sync();
            const uint32_t a = smem_addr(sm + s * kStage), b = a + A_BYTES;
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              if constexpr (PAIR)
                tc::mma_bf16_pair(d, tc::desc_kmajor_sw128(a + k * 32), tc::desc_kmajor_sw128(b + k * 32), idesc,
                                  (kb | k) != 0);
              else
                tc::mma_bf16(d, tc::desc_kmajor_sw128(a + k * 32), tc::desc_kmajor_sw128(b + k * 32), idesc,
                             (kb | k) != 0);
            }
            if constexpr (PAIR) tc::mma_commit_pair(&empty[s], 0x3);
            else tc::mma_commit(&empty[s]);
          }
          if (ok) {
            if constexpr (PAIR) tc::mma_commit_pair(&accf[acc], 0x3);
            else tc::mma_commit(&accf[acc]);
          }
        }
      }
    }
  } else {
    // ---------------------------------------------------------------- epilogue (4 warps)
    const int q = warp & 3;  // TMEM lane quarter this warp may access
    const int rl = 32 * q + lane;
    const float kNegInf = -__int_as_float(0x7f800000);
    uint32_t t = 0;
    bool ok = true;
    for (int item = unit; item < n_items && ok; item += n_units) {
      const int vb = item / n_m, m0 = (item % n_m) * kMStep + static_cast<int>(rank) * BM;
      const int r = m0 + rl;  // token within the chunk
      const bool row_ok = r < ch.count;
      const int nt1 = min((vb + 1) * p.vb_tiles, p.n_nt);
      // running partials of the block's even and odd tiles (the halves of its 256 x 512 tiles);
      // with TILE_PARTS the tiles' own go out
      SoftmaxPartial ps0{kNegInf, 0.f, 0.f}, ps1{kNegInf, 0.f, 0.f};
      float za = 0.f;
      const int32_t a = row_ok ? p.token_ids[token_of(p.tok, ch, r)] : -1;
      for (int nt = vb * p.vb_tiles; nt < nt1; ++nt, ++t) {
        const int acc = t & 1;
        if (!mbar_wait_bounded(&accf[acc], (t >> 1) & 1)) {
          if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const int n0 = nt * BN;
        const uint32_t tbase_acc = tmem + (static_cast<uint32_t>(32 * q) << 16) + acc * BN;
        // sweep 1: the tile's row maximum and the sampled id's logit
        float tm = kNegInf;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          const int col0 = n0 + c;
          const int nvalid = min(32, p.V - col0);
          if (nvalid <= 0) break;  // past the vocabulary (uniform across the warp)
          float v[32];
          tc::tmem_ld32(tbase_acc + c, v);
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (j < nvalid) tm = fmaxf(tm, v[j]);
          const int ja = a - col0;
          if (ja >= 0 && ja < 32) {
#pragma unroll
            for (int j = 0; j < 32; ++j)
              if (j == ja) za = v[j];
          }
        }
        // sweep 2: e = exp(z - m_j), its sums, and (STATS_P) e stored in bf16
        const float nm = -tm * kLog2e;
        float s0 = 0.f, s1 = 0.f, u0 = 0.f;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          const int col0 = n0 + c;
          const int nvalid = min(32, p.V - col0);
          if (nvalid <= 0) break;
          float v[32];
          tc::tmem_ld32(tbase_acc + c, v);
          uint32_t w[16];
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            float e2[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const bool in = j + h < nvalid;
              const float z = in ? v[j + h] : tm;
              const float e = in ? ex2(fmaf(z, kLog2e, nm)) : 0.f;
              if (h) s1 += e; else s0 += e;
              if (p.ent) u0 = fmaf(e, z - tm, u0);
              e2[h] = e;
            }
            w[j / 2] = pack_bf16x2(e2[0], e2[1]);
          }
          if (MODE == STATS_P && row_ok) {
            uint16_t* out = p.dz + static_cast<int64_t>(ch.row + r) * p.ldz + col0;
            if (nvalid == 32) {
#pragma unroll
              for (int j = 0; j < 4; ++j)
                *reinterpret_cast<uint4*>(out + 8 * j) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
            } else {
#pragma unroll
              for (int j = 0; j < 32; ++j)
                if (j < nvalid) out[j] = static_cast<uint16_t>((w[j / 2] >> (16 * (j & 1))) & 0xFFFFu);
            }
          }
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) {
          if (PAIR && rank != 0) mbar_arrive_remote(map_to_rank(smem_addr(&acce[acc]), 0));
          else mbar_arrive(&acce[acc]);
        }
        if (MODE == STATS_P && row_ok) p.tmax[static_cast<int64_t>(r) * p.n_nt + nt] = tm;
        const SoftmaxPartial tile{tm, s0 + s1, u0};
        if (TILE_PARTS) {
          if (row_ok) p.partials[static_cast<int64_t>(nt) * p.tok.Tc + r] = make_float4(tile.m, tile.s, tile.u, za);
          za = 0.f;
        } else if (nt & 1) {
          ps1 = merge(ps1, tile);
        } else {
          ps0 = merge(ps0, tile);
        }
      }
      if (ok && row_ok && !TILE_PARTS) {
        p.partials[static_cast<int64_t>(2 * vb) * p.tok.Tc + r] = make_float4(ps0.m, ps0.s, ps0.u, za);
        p.partials[static_cast<int64_t>(2 * vb + 1) * p.tok.Tc + r] = make_float4(ps1.m, ps1.s, ps1.u, 0.f);
      }
    }
  }
  tc::fence_before_sync();
  if constexpr (PAIR) cluster_sync_all();
  else __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    if constexpr (PAIR) tc::tmem_dealloc_pair(tmem, 2 * BN);
    else tc::tmem_dealloc(tmem, 2 * BN);
  }
}

// ------------------------------------------------------------------ 256 x 512 tiles
//
// Wide form of the pair kernel: a CTA pair computes 256 tokens x 512 vocabulary entries per
// tile with two cta_group::2 MMAs per K step that share the H operand, into one accumulator of
// all 512 TMEM columns (4 stages of 48 KB: this CTA's 128 tokens of H and, per MMA, its 128
// of the 256 W rows). The epilogue treats the tile as two 256-column halves with the same two
// sweeps as the 256 x 256 form (so the tile maxima keep their 256-column granularity), one
// group of four warps per half, each with its own partial (the block's even or odd tiles, as
// in the 256 x 256 form, so both forms give the same bits). It cannot overlap the next
// tile's MMAs: the single accumulator is handed back after both halves; the second group
// halves the time that takes.
constexpr uint32_t W_HALF = (BN / 2) * BK * 2;          // 16 KB
constexpr uint32_t STAGEW_BYTES = A_BYTES + 2 * W_HALF;  // 48 KB
constexpr int NSW = 4;
constexpr size_t kSmemW = NSW * STAGEW_BYTES + 1024;

// One 256-column half of a tile's epilogue: the row maximum of the valid columns and the
// sampled id's logit (za), then e = exp(z - m), its sums and (STATS_P) e in bf16 at `out`.
template <int MODE>
__device__ __forceinline__ SoftmaxPartial epi_half(uint32_t tacc, int n0, int V, int32_t a, int ent, uint16_t* out,
                                                   float& za, float& tm_out) {
  const float kNegInf = -__int_as_float(0x7f800000);
  float tm = kNegInf;
#pragma unroll 1
  for (int c = 0; c < BN; c += 32) {
    const int col0 = n0 + c;
    const int nvalid = min(32, V - col0);
    if (nvalid <= 0) break;  // past the vocabulary (uniform across the warp)
    float v[32];
    tc::tmem_ld32(tacc + c, v);
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < nvalid) tm = fmaxf(tm, v[j]);
    const int ja = a - col0;
    if (ja >= 0 && ja < 32) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (j == ja) za = v[j];
    }
  }
  const float nm = -tm * kLog2e;
  float s0 = 0.f, s1 = 0.f, u0 = 0.f;
#pragma unroll 1
  for (int c = 0; c < BN; c += 32) {
    const int col0 = n0 + c;
    const int nvalid = min(32, V - col0);
    if (nvalid <= 0) break;
    float v[32];
    tc::tmem_ld32(tacc + c, v);
    uint32_t w[16];
#pragma unroll
    for (int j = 0; j < 32; j += 2) {
      float e2[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool in = j + h < nvalid;
        const float z = in ? v[j + h] : tm;
        const float e = in ? ex2(fmaf(z, kLog2e, nm)) : 0.f;
        if (h) s1 += e; else s0 += e;
        if (ent) u0 = fmaf(e, z - tm, u0);
        e2[h] = e;
      }
      w[j / 2] = pack_bf16x2(e2[0], e2[1]);
    }
    if (MODE == STATS_P && out) {
      uint16_t* o = out + c;
      if (nvalid == 32) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<uint4*>(o + 8 * j) = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      } else {
#pragma unroll
        for (int j = 0; j < 32; ++j)
          if (j < nvalid) o[j] = static_cast<uint16_t>((w[j / 2] >> (16 * (j & 1))) & 0xFFFFu);
      }
    }
  }
  tm_out = tm;
  return SoftmaxPartial{tm, s0 + s1, u0};
}

// warp 0 TMA, warp 1 MMA, warps 2-9 epilogue: warps 2-5 read the tile's first 256 columns and
// warps 6-9 its second 256, each group with its own running partial (two per vocabulary block)
constexpr int kThreadsW = 320;

template <int MODE, bool TILE_PARTS>
__global__ void __launch_bounds__(kThreadsW, 1) head_wide_kernel(const __grid_constant__ CUtensorMap tmH,
                                                                const __grid_constant__ CUtensorMap tmW,
                                                                const HeadArgs p) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[NSW], empty[NSW], accf, acce;
  __shared__ uint32_t tbase;
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int unit = static_cast<int>(blockIdx.x >> 1);
  const int n_units = static_cast<int>(gridDim.x >> 1);
  const int VB2 = p.vb_tiles / 2;  // 512-column tiles per vocabulary block
  const Chunk ch = chunk_of(p.tok, p.chunk);
  const int n_m = (ch.count + 2 * BM - 1) / (2 * BM);
  const int n_nt2 = (p.n_nt + 1) / 2;
  const int n_items = n_m * p.n_vb;
  const int nkb = p.D / BK;
  if (n_items == 0) return;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSW; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accf, 1);
    mbar_init(&acce, 16);  // 8 epilogue warps in each CTA of the pair
    fence_mbar_init();
  }
  if (warp == 1) tc::tmem_alloc_pair(&tbase, 2 * BN);
  tc::fence_before_sync();
  cluster_sync_all();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;

  if (warp == 0) {
    if (lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      for (int item = unit; item < n_items && ok; item += n_units) {
        const int vb = item / n_m, m0 = (item % n_m) * 2 * BM + static_cast<int>(rank) * BM;
        const int nt1 = min((vb + 1) * VB2, n_nt2);
        for (int nt = vb * VB2; nt < nt1 && ok; ++nt) {
          for (int kb = 0; kb < nkb; ++kb, ++g) {
            const int s = g % NSW;
            const uint32_t use = g / NSW;
            if (use > 0 && !mbar_wait_bounded(&empty[s], (use - 1) & 1)) {
              flag_status(p.status, RL_DEV_TIMEOUT);
              ok = false;
              break;
            }
            uint8_t* st = sm + s * STAGEW_BYTES;
            if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * STAGEW_BYTES);  // both CTAs' bytes
            const uint32_t bar = map_to_rank(smem_addr(&full[s]), 0);
            tc::tma_load_2d_pair(st, &tmH, kb * BK, ch.row + m0, bar);
#pragma unroll
            for (int h = 0; h < 2; ++h)
              tc::tma_load_2d_pair(st + A_BYTES + h * W_HALF, &tmW, kb * BK,
                                   nt * 2 * BN + h * BN + static_cast<int>(rank) * (BN / 2), bar);
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = tc::idesc_bf16_f32(2 * BM, BN);
      uint32_t g = 0, t = 0;
      bool ok = true;
      for (int item = unit; item < n_items && ok; item += n_units) {
        const int vb = item / n_m;
        const int nt1 = min((vb + 1) * VB2, n_nt2);
        for (int nt = vb * VB2; nt < nt1 && ok; ++nt, ++t) {
          if (t > 0 && !mbar_wait_cluster_bounded(&acce, (t - 1) & 1)) {
            flag_status(p.status, RL_DEV_TIMEOUT);
            ok = false;
            break;
          }
          tc::fence_after_sync();
          for (int kb = 0; kb < nkb; ++kb, ++g) {
            const int s = g % NSW;
            if (!mbar_wait_bounded(&full[s], (g / NSW) & 1)) {
              flag_status(p.status, RL_DEV_TIMEOUT);
              ok = false;
              break;
            }
            tc::fence_after_sync();
            const uint32_t a = smem_addr(sm + s * STAGEW_BYTES), b = a + A_BYTES;
#pragma unroll
            for (int k = 0; k < BK / 16; ++k) {
              const uint64_t ad = tc::desc_kmajor_sw128(a + k * 32);
#pragma unroll
              for (int h = 0; h < 2; ++h)
                tc::mma_bf16_pair(tmem + h * BN, ad, tc::desc_kmajor_sw128(b + h * W_HALF + k * 32), idesc,
                                  (kb | k) != 0);
            }
            tc::mma_commit_pair(&empty[s], 0x3);
          }
          if (ok) tc::mma_commit_pair(&accf, 0x3);
        }
      }
    }
  } else {
    const int q = warp & 3;            // TMEM lane quarter this warp may access
    const int h = (warp - 2) >> 2;     // the 256-column half of each tile this warp reads
    const int rl = 32 * q + lane;
    const float kNegInf = -__int_as_float(0x7f800000);
    const uint32_t tq = tmem + (static_cast<uint32_t>(32 * q) << 16);
    uint32_t t = 0;
    bool ok = true;
    for (int item = unit; item < n_items && ok; item += n_units) {
      const int vb = item / n_m, m0 = (item % n_m) * 2 * BM + static_cast<int>(rank) * BM;
      const int r = m0 + rl;
      const bool row_ok = r < ch.count;
      const int nt1 = min((vb + 1) * VB2, n_nt2);
      SoftmaxPartial ps{kNegInf, 0.f, 0.f};
      float za = 0.f;
      const int32_t a = row_ok ? p.token_ids[token_of(p.tok, ch, r)] : -1;
      uint16_t* dz_row = (MODE == STATS_P && row_ok) ? p.dz + static_cast<int64_t>(ch.row + r) * p.ldz : nullptr;
      for (int nt = vb * VB2; nt < nt1; ++nt, ++t) {
        if (!mbar_wait_sleep_bounded(&accf, t & 1)) {
          if (lane == 0) flag_status(p.status, RL_DEV_TIMEOUT);
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const int j = nt * 2 + h;  // 256-column tile
        if (j < p.n_nt) {
          float tm;
          const SoftmaxPartial half =
              epi_half<MODE>(tq + h * BN, j * BN, p.V, a, p.ent, dz_row ? dz_row + j * BN : nullptr, za, tm);
          if (MODE == STATS_P && row_ok) p.tmax[static_cast<int64_t>(r) * p.n_nt + j] = tm;
          if (TILE_PARTS) {
            if (row_ok) p.partials[static_cast<int64_t>(j) * p.tok.Tc + r] = make_float4(half.m, half.s, half.u, za);
            za = 0.f;
          } else {
            ps = merge(ps, half);
          }
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) {
          if (rank != 0) mbar_arrive_remote(map_to_rank(smem_addr(&acce), 0));
          else mbar_arrive(&acce);
        }
      }
      if (ok && row_ok && !TILE_PARTS)
        p.partials[static_cast<int64_t>(2 * vb + h) * p.tok.Tc + r] = make_float4(ps.m, ps.s, ps.u, za);
    }
  }
  tc::fence_before_sync();
  cluster_sync_all();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc_pair(tmem, 2 * BN);
  }
}

struct DzArgs {
  Tokens tok;
  int32_t chunk;
  int32_t V, n_nt, n_traj;
  int32_t n_part, n_tile;           // block partials per token; tile partials, or 0: see merge_partials
  int32_t split;                    // CTAs per row
  int32_t ent;                      // the entropy term is in the gradient
  const float4* partials;
  const float* tmax;                // [Tc x n_nt]
  uint16_t* dz;                     // in: e = exp(z - m_j) (bf16); out: dZ (bf16)
  int64_t ldz;
  const int32_t* token_ids;
  const uint8_t* mask;
  const int32_t* token_traj;
  const float* adv;
  const float* coef;
  const float* old_logp;
  const float* ref_logp;
  const float* rollout_logp;
  float clip_lo, clip_hi, beta, alpha, tis_cap;
  int32_t adv_per_row;  // adv holds one A_t per token (else one per trajectory)
  double* row_loss;     // [T]
  uint32_t* counter;    // the products' work counter, set back here for their next launch
  float* token_stats;
  int32_t* status;
};

// A token's partials (`stride` apart), merged by a warp: lane l takes the block partials l, l + 32, ... in
// order, the lanes are combined by shuffles (in head_dz_kernel and in head_logp_merge_kernel: the loss
// call and the forward-only call give the same bits). Where the statistics pass left every tile's own
// (n_tile of them, else 0), a block's partial is formed here first, tile by tile as the pass would, with
// LOADS of them in flight. A thread per token walking them 8 loads at a time took 16 us for 4,096 tokens,
// a warp 6.
template <int LOADS>
__device__ __forceinline__ void merge_partials(const float4* partials, int64_t stride, int n_part, int n_tile,
                                               SoftmaxPartial& q, float& za) {
  const int lane = threadIdx.x & 31;
  if (n_tile == 0) {
#pragma unroll 4
    for (int b = lane; b < n_part; b += 32) {
      const float4 w = partials[b * stride];
      q = merge(q, SoftmaxPartial{w.x, w.y, w.z});
      za += w.w;  // nonzero in the one partial whose columns hold the sampled id
    }
  } else {
    for (int b = lane; b < n_part; b += 32) {
      const int first = (b >> 1) * kMaxVb + (b & 1);
      SoftmaxPartial blk{-__int_as_float(0x7f800000), 0.f, 0.f};
#pragma unroll
      for (int h = 0; h < kMaxVb; h += 2 * LOADS) {
        float4 w[LOADS];
#pragma unroll
        for (int k = 0; k < LOADS; ++k) {
          const int nt = first + h + 2 * k;
          if (nt < n_tile) w[k] = partials[nt * stride];
        }
#pragma unroll
        for (int k = 0; k < LOADS; ++k) {
          if (first + h + 2 * k >= n_tile) break;
          blk = merge(blk, SoftmaxPartial{w[k].x, w[k].y, w[k].z});
          za += w[k].w;
        }
      }
      q = merge(q, blk);
    }
  }
  q = warp_merge<true>(q);
  za = warp_sum(za);
}

constexpr int kMergeThreads = 128;
constexpr int kMergeRows = kMergeThreads / 32;

// Row r's coefficients, by one warp (the same in every lane): the vocabulary blocks' partials merged
// in a fixed order and the per-token objective terms. With `write` lane 0 also writes the token's
// loss contribution and statistics. The words that need only the token are loaded together.
__device__ __forceinline__ RowCoef row_coef(const DzArgs& p, const Chunk& ch, int r, const float4* partials, int64_t stride,
                                            bool write) {
  const int64_t t = token_of(p.tok, ch, r);
  const uint8_t m = p.mask[t];
  const int32_t i = p.token_traj[t], a = p.token_ids[t];
  const float old = p.old_logp[t];
  const float ref = p.ref_logp ? p.ref_logp[t] : 0.f;
  const float roll = p.rollout_logp ? p.rollout_logp[t] : 0.f;
  SoftmaxPartial q{-__int_as_float(0x7f800000), 0.f, 0.f};
  float za = 0.f;
  merge_partials<4>(partials, stride, p.n_part, p.n_tile, q, za);
  write = write && (threadIdx.x & 31) == 0;
  RowCoef rc = {};
  rc.a = -1;
  bool active = m != 0;
  float c = 0.f, A = 0.f;
  if (active) {
    if (i < 0 || i >= p.n_traj) {
      if (write) flag_status(p.status, RL_DEV_BAD_TRAJ);
      active = false;
    } else {
      c = p.coef[i];
      A = p.adv_per_row ? p.adv[t] : p.adv[i];
      active = c != 0.f;
    }
  }
  if (active && (a < 0 || a >= p.V)) {
    if (write) flag_status(p.status, RL_DEV_BAD_TOKEN);
    active = false;
  }
  if (!active) {
    if (write) {
      p.row_loss[t] = 0.0;
      if (p.token_stats)
        for (int k = 0; k < 5; ++k) p.token_stats[t * 5 + k] = 0.f;
    }
    return rc;
  }
  const float lnS = logf(q.s);
  const float lse = q.m + lnS;
  const float H = lnS - q.u / q.s;
  const float logp = za - lse;
  const float rho = expf((za - old) - lse);
  const float crho = fminf(fmaxf(rho, p.clip_lo), p.clip_hi);
  const float surr = fminf(rho * A, crho * A);
  const bool cut = (A > 0.f && rho > p.clip_hi) || (A < 0.f && rho < p.clip_lo);
  const float w = (p.tis_cap > 0.f && p.rollout_logp) ? fminf(expf(old - roll), p.tis_cap) : 1.f;
  float kl = 0.f, dkl = 0.f;
  if (p.beta != 0.f && p.ref_logp) {
    const float d = (ref - za) + lse;
    const float ed = expf(d);
    kl = ed - d - 1.f;
    dkl = 1.f - ed;
  }
  const float ell = -w * surr + p.beta * kl - p.alpha * H;
  const float g = (cut ? 0.f : -w * A * rho) + p.beta * dkl;
  const float cg = c * g, ca = c * p.alpha;
  rc.nlse2 = -lse * kLog2e;
  rc.Kp = -cg;
  rc.cg = cg;
  rc.ca = ca;
  rc.Ke = -cg + ca * (H - lse);
  rc.a = a;
  rc.active = 1;
  if (write) {
    p.row_loss[t] = static_cast<double>(c) * static_cast<double>(ell);
    if (p.token_stats) {
      float* st = p.token_stats + t * 5;
      st[0] = logp; st[1] = rho; st[2] = cut ? 1.f : 0.f; st[3] = H; st[4] = kl;
    }
  }
  return rc;
}

constexpr int kDzThreads = 256;
constexpr int kDzLoads = 4;          // vectors in flight per thread
constexpr int kTilesStaged = 640;    // tile partials of a row staged in shared memory: V up to 163,840
constexpr int kMaxTilesSmem = 2048;  // V up to 524,288 keeps the row's tile factors in shared memory

// p.split CTAs per token row of the chunk (grid-stride): the CTA's first warp merges the row's
// partials into its coefficients while the others' first loads are on their way, then
// p_v = e_v exp(m_j - lse) and dZ_v = Kp p_v (+ cg at v = a), or with the entropy bonus
// p_v (ca z_v + Ke) (+ cg at v = a), z_v = m_j + ln e_v. Rows that are not trained on become zeros.
// 16-byte loads and stores.
//
// HBM bounds it in a full chunk (2 x 2 B per logit), the chain of trips to memory in a short call: the
// merge, the rescale and the reset of the products' counter were three launches of 7, 14 and 2 us
// at 500 tokens x 32,000 entries with one CTA and one vector in flight per thread and row; this one
// takes 15 (serialised, cold caches).
__global__ void __launch_bounds__(kDzThreads, 4) head_dz_kernel(const DzArgs p) {
  __shared__ float fac[kMaxTilesSmem], zoff[kMaxTilesSmem];
  __shared__ RowCoef shared_rc;
  __shared__ float4 tiles[kTilesStaged];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Chunk ch = chunk_of(p.tok, p.chunk);
  if (blockIdx.x == 0 && tid == 0) *p.counter = 0u;
  const int nvec = p.V / 8, split = p.split;
  for (int item = blockIdx.x; item < ch.padded * split; item += gridDim.x) {
    const int r = item / split, part = item - r * split;
    uint16_t* row = p.dz + static_cast<int64_t>(ch.row + r) * p.ldz;
    uint4* vec = reinterpret_cast<uint4*>(row);
    // the CTA's vectors (and, in the row's last part, the elements after them), and their tiles
    const int k_lo = static_cast<int>(static_cast<int64_t>(nvec) * part / split);
    const int k_hi = static_cast<int>(static_cast<int64_t>(nvec) * (part + 1) / split);
    const int tail = part == split - 1 ? nvec * 8 : p.V;
    if (r >= ch.count) {  // rows past the chunk's tokens: zeros
      for (int k = k_lo + tid; k < k_hi; k += kDzThreads) vec[k] = make_uint4(0, 0, 0, 0);
      for (int v = tail + tid; v < p.V; v += kDzThreads) row[v] = 0;
      continue;
    }
    const int j_lo = k_lo * 8 / BN, j_hi = part == split - 1 ? p.n_nt : (k_hi * 8 + BN - 1) / BN;
    uint4 w[kDzLoads];
    auto load = [&](int k0) {
#pragma unroll
      for (int i = 0; i < kDzLoads; ++i) {
        const int k = k0 + i * kDzThreads;
        if (k < k_hi) w[i] = vec[k];
      }
    };
    load(k_lo + tid);
    float m = j_lo + tid < j_hi ? p.tmax[static_cast<int64_t>(r) * p.n_nt + j_lo + tid] : 0.f;
    // a short call's tile partials come in one trip of the whole CTA
    const bool staged = p.n_tile != 0 && p.n_tile <= kTilesStaged;
    if (staged) {
      for (int t = tid; t < p.n_tile; t += kDzThreads) tiles[t] = p.partials[static_cast<int64_t>(t) * p.tok.Tc + r];
      __syncthreads();
    }
    if (warp == 0) {
      const RowCoef c = row_coef(p, ch, r, staged ? tiles : p.partials + r, staged ? 1 : p.tok.Tc, part == 0);
      if (lane == 0) shared_rc = c;
    }
    __syncthreads();
    const RowCoef rc = shared_rc;
    // per tile: Kp exp(m_j - lse) (no entropy) or exp(m_j - lse) and m_j (entropy)
    for (int j = j_lo + tid; j < j_hi; j += kDzThreads) {
      if (j >= j_lo + kDzThreads) m = p.tmax[static_cast<int64_t>(r) * p.n_nt + j];
      const float f = ex2(fmaf(m, kLog2e, rc.nlse2));
      fac[j] = p.ent ? f : rc.Kp * f;
      zoff[j] = fmaf(rc.ca, m, rc.Ke);  // ca m_j + Ke
    }
    __syncthreads();
    if (!rc.active) {
      for (int k = k_lo + tid; k < k_hi; k += kDzThreads) vec[k] = make_uint4(0, 0, 0, 0);
      for (int v = tail + tid; v < p.V; v += kDzThreads) row[v] = 0;
      continue;
    }
    for (int k0 = k_lo + tid; k0 < k_hi; k0 += kDzLoads * kDzThreads) {
      if (k0 != k_lo + tid) load(k0);
#pragma unroll
      for (int i = 0; i < kDzLoads; ++i) {
        const int k = k0 + i * kDzThreads;
        if (k >= k_hi) break;
        const int j = (k * 8) / BN;
        const float f = fac[j];
        uint32_t wp[4] = {w[i].x, w[i].y, w[i].z, w[i].w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          float o[2];
#pragma unroll
          for (int b = 0; b < 2; ++b) {
            const float e = b ? bf16_hi(wp[h]) : bf16_lo(wp[h]);
            float x;
            if (p.ent) {
              // p (ca z + Ke) with z = m_j + ln e; e = 0 contributes 0
              x = e > 0.f ? f * e * fmaf(rc.ca, __logf(e), zoff[j]) : 0.f;
            } else {
              x = f * e;
            }
            if (k * 8 + 2 * h + b == rc.a) x += rc.cg;
            o[b] = x;
          }
          wp[h] = pack_bf16x2(o[0], o[1]);
        }
        vec[k] = make_uint4(wp[0], wp[1], wp[2], wp[3]);
      }
    }
    for (int v = tail + tid; v < p.V; v += kDzThreads) {
      const int j = v / BN;
      const float e = bf16_to_f32(row[v]);
      float x = p.ent ? (e > 0.f ? fac[j] * e * fmaf(rc.ca, __logf(e), zoff[j]) : 0.f) : fac[j] * e;
      if (v == rc.a) x += rc.cg;
      row[v] = f32_to_bf16(x);
    }
    // the next row's shared_rc and tiles are written past this row's last barrier, its fac and zoff past
    // the next row's first: every read of this row's comes before
  }
}

struct LogpMergeArgs {
  Tokens tok;
  int32_t chunk;
  int32_t V, n_part, n_tile;  // as in DzArgs
  const float4* partials;
  const int32_t* token_ids;
  float* logp_out;
  float* entropy_out;
  float* lse_out;
  int32_t* status;
};

// Forward-only merge: one warp per token of the chunk writes logp, H and lse.
__global__ void __launch_bounds__(kMergeThreads) head_logp_merge_kernel(const LogpMergeArgs p) {
  const int r = static_cast<int>(blockIdx.x) * kMergeRows + static_cast<int>(threadIdx.x >> 5);
  const bool lead = (threadIdx.x & 31) == 0;
  const Chunk ch = chunk_of(p.tok, p.chunk);
  if (r >= ch.count) return;
  const int64_t t = token_of(p.tok, ch, r);
  SoftmaxPartial q{-__int_as_float(0x7f800000), 0.f, 0.f};
  float za = 0.f;
  merge_partials<8>(p.partials + r, p.tok.Tc, p.n_part, p.n_tile, q, za);
  if (!lead) return;
  const float lnS = logf(q.s);
  const float lse = q.m + lnS;
  const int32_t a = p.token_ids[t];
  const bool a_ok = a >= 0 && a < p.V;
  if (!a_ok) flag_status(p.status, RL_DEV_BAD_TOKEN);
  p.logp_out[t] = a_ok ? za - lse : __int_as_float(0x7fc00000);
  if (p.entropy_out) p.entropy_out[t] = lnS - q.u / q.s;
  if (p.lse_out) p.lse_out[t] = lse;
}

// ------------------------------------------------------------------ trained tokens
//
// A token that is not trained on (M_t = 0, c = 0, or a bad id or owner, which is flagged) has no
// loss and a zero gradient, so it needs none of the three products: head_select_kernel (after
// head_count_kernel in a call of more than 8,192 tokens) lists the
// trained tokens in their order (and the others from the list's end), head_gather_kernel packs a
// chunk's hidden states, and everything after it works on packed rows. On the multi-turn batch
// (62% trained) that is 38% of the call's flops: 6,000 tokens at D = 4,096 and V = 151,936
// 14.2 -> 11.1 ms (13.9 -> 9.3 to 10.7 ms in other runs: power, and how many tokens are trained).
struct SelectArgs {
  int32_t T, V, n_traj;
  const int32_t* token_ids;
  const uint8_t* mask;
  const int32_t* token_traj;
  const float* coef;
  int32_t* idx;      // [T]
  int32_t* n_dev;    // number of trained tokens
  int32_t* counts;   // per kSelThreads tokens, from head_count_kernel; null: a short call, without it
  double* row_loss;  // 0 for the others
  float* token_stats;
  int32_t* status;
};

constexpr int kSelThreads = 1024;
// CTAs of head_select_kernel up to which it counts by itself.
constexpr int64_t kSelAlone = 8;
static int64_t select_blocks(int64_t T) { return (T + kSelThreads - 1) / kSelThreads; }

__device__ __forceinline__ bool is_trained(const SelectArgs& p, int64_t t, bool flag) {
  if (p.mask[t] == 0) return false;
  const int32_t i = p.token_traj[t];
  if (i < 0 || i >= p.n_traj) {
    if (flag) flag_status(p.status, RL_DEV_BAD_TRAJ);
    return false;
  }
  if (p.coef[i] == 0.f) return false;
  const int32_t a = p.token_ids[t];
  if (a < 0 || a >= p.V) {
    if (flag) flag_status(p.status, RL_DEV_BAD_TOKEN);
    return false;
  }
  return true;
}

// Trained tokens of each kSelThreads tokens.
__global__ void __launch_bounds__(kSelThreads) head_count_kernel(const SelectArgs p) {
  const int64_t t = static_cast<int64_t>(blockIdx.x) * kSelThreads + threadIdx.x;
  const int n = __syncthreads_count(t < p.T && is_trained(p, t, false));
  if (threadIdx.x == 0) p.counts[blockIdx.x] = n;
}

// One CTA per kSelThreads tokens. The trained tokens before its own: the earlier CTAs' counts, or, in a
// short call, counted here, which spares a launch but reads every earlier token again: 5 us for 4,096
// tokens, 7 for 8,192, 11 for 16,384, 18 for 32,768 and 386 for 524,288, against 6 (16,384 and
// 32,768) and 13 us for the two launches.
__global__ void __launch_bounds__(kSelThreads) head_select_kernel(const SelectArgs p) {
  __shared__ int32_t part[kSelThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * kSelThreads, t = t0 + tid;
  int32_t before = 0;
  if (p.counts) {
    for (unsigned b = tid; b < blockIdx.x; b += kSelThreads) before += p.counts[b];
  } else {
#pragma unroll 4
    for (int64_t u = tid; u < t0; u += kSelThreads) before += is_trained(p, u, false) ? 1 : 0;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  if (lane == 0) part[warp] = before;
  __syncthreads();
  int32_t base = 0;
  for (int w = 0; w < kSelThreads / 32; ++w) base += part[w];
  __syncthreads();
  const bool on = t < p.T && is_trained(p, t, true);
  const unsigned ballot = __ballot_sync(0xffffffffu, on);
  if (lane == 0) part[warp] = __popc(ballot);
  __syncthreads();
  int32_t rank = base + __popc(ballot & ((1u << lane) - 1u)), all = base;
  for (int w = 0; w < kSelThreads / 32; ++w) {
    if (w < warp) rank += part[w];
    all += part[w];
  }
  if (t < p.T) {
    if (on) {
      p.idx[rank] = static_cast<int32_t>(t);
    } else {
      p.idx[p.T - 1 - (t - rank)] = static_cast<int32_t>(t);  // t - rank untrained tokens before it
      p.row_loss[t] = 0.0;
      if (p.token_stats)
        for (int k = 0; k < 5; ++k) p.token_stats[t * 5 + k] = 0.f;
    }
  }
  if (blockIdx.x == gridDim.x - 1 && tid == 0) *p.n_dev = all;
}

struct GatherArgs {
  Tokens tok;
  int32_t chunk;
  int32_t D;            // a multiple of 64
  int32_t dh_bytes;     // bytes per element of d_hidden
  const uint16_t* hidden;
  uint16_t* packed;     // [G Tc x D]
  char* d_hidden;
};

// Packs the hidden states of the chunk's tokens (zeros up to `padded`, where the product over
// tokens reads whole blocks of 64); the first chunk's launch also writes the zero d_hidden rows of
// the tokens that are not trained on. A warp per row, 16 bytes per lane and access.
__global__ void __launch_bounds__(256) head_gather_kernel(const GatherArgs p) {
  const int lane = threadIdx.x & 31;
  const Chunk ch = chunk_of(p.tok, p.chunk);
  const int64_t warps = static_cast<int64_t>(gridDim.x) * 8;
  const int vec = p.D / 8;
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5); r < ch.padded; r += warps) {
    uint4* dst = reinterpret_cast<uint4*>(p.packed + (ch.row + r) * p.D);
    if (r < ch.count) {
      const uint4* src = reinterpret_cast<const uint4*>(p.hidden + static_cast<int64_t>(token_of(p.tok, ch, r)) * p.D);
#pragma unroll 8
      for (int k = lane; k < vec; k += 32) dst[k] = src[k];
    } else {
      for (int k = lane; k < vec; k += 32) dst[k] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
  if (p.chunk != 0) return;
  const int64_t row16 = static_cast<int64_t>(p.D) * p.dh_bytes / 16;
  for (int64_t k = *p.tok.n_dev + static_cast<int64_t>(blockIdx.x) * 8 + (threadIdx.x >> 5); k < p.tok.T; k += warps) {
    uint4* row = reinterpret_cast<uint4*>(p.d_hidden) + p.tok.idx[k] * row16;
    for (int64_t q = lane; q < row16; q += 32) row[q] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// ------------------------------------------------------------------ host side

// bf16 matrix [rows x inner] (row stride inner), tiles of box_rows x 64 with the 128-byte swizzle.
static rl_status make_map(CUtensorMap* m, const void* base, int64_t inner, int64_t rows, uint32_t box_rows) {
  return tmap_2d(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, base, inner, rows, inner * 2, 64, box_rows,
                 CU_TENSOR_MAP_SWIZZLE_128B);
}

// N tiles per work item of the statistics pass. Items are 256 tokens x a block of the vocabulary;
// blocks of 16 tiles leave few partials, but a short chunk then has fewer items than CTA pairs (500
// tokens x 32,000 entries: 16 items on 76 pairs, 121 us). The largest of 16, 8, 4 and 2 tiles
// whose longest pair does at most 3% more tiles than the best of them: full chunks keep 16. The
// split changes no token's statistics: see merge_partials.
static int64_t vb_tiles(int64_t Tc, int64_t n_nt) {
  const int64_t n_m = (Tc + 2 * BM - 1) / (2 * BM);
  auto cost = [&](int64_t vb) { return (n_m * ((n_nt + vb - 1) / vb) + kPairs - 1) / kPairs * vb; };
  const int64_t best = std::min(std::min(cost(16), cost(8)), std::min(cost(4), cost(2)));
  for (int64_t vb = kMaxVb; vb > 2; vb /= 2)
    if (100 * cost(vb) <= 103 * best) return vb;
  return 2;
}

// Parts of the contraction over V in dH = dZ W. A dH tile is 256 tokens x 512 columns over the
// whole vocabulary, by far the longest item of the backward launch: with fewer than half as many
// of them as CTA pairs they outlast everything else (500 tokens, D = 1,024: 4 tiles, 285 us), so
// each is cut into parts whose fp32 sums head_combine_kernel adds in order.
static int64_t dh_parts(int64_t Tc, int64_t V, int64_t D) {
  const int64_t tiles = (Tc + 2 * BM - 1) / (2 * BM) * ((D + 511) / 512);
  if (2 * tiles >= kPairs) return 1;
  const int64_t most = std::max<int64_t>(1, V / 1024);  // at least 16 K blocks of 64 per part
  return std::min(std::min<int64_t>(16, most), (kPairs + tiles - 1) / tiles);
}

// CTAs that share a row of the rescale: as many as give every SM eight CTAs, down to 512 vectors
// (two per thread) each; one where the chunk's rows suffice.
static int dz_split(int64_t Tc, int64_t V) {
  const int64_t most = std::max<int64_t>(1, V / 8 / 512);
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>(most, 152 * 8 / Tc)));
}

struct Layout {
  int64_t Tc, G, n_nt, n_vb, ldz;  // G chunks per group
  int64_t vb, parts;               // N tiles per work item; parts of dH's contraction
  int64_t n_part;                  // partials of blocks of 16 tiles (two each)
  bool tile_parts;                 // the workspace holds every tile's partial instead
  bool pack;                       // the trained tokens are packed
  size_t off_partials, off_tmax, off_idx, off_counts, off_h, off_parts, off_dz, total;
};

static size_t al256(size_t x) { return (x + 255) & ~size_t(255); }

// The softmax partials of one chunk.
static size_t partials_bytes(const Layout& L) {
  return al256(static_cast<size_t>((L.tile_parts ? L.n_nt : L.n_part) * L.Tc) * sizeof(float4));
}

// What a workspace has room for: only what every call needs (every token goes through the products,
// work items of 16 tiles); the packed trained tokens and the tiles' partials besides; and the
// parts of dH besides.
enum Room { kLeast = 0, kPacked = 1, kAll = 2 };

// Workspace of the loss call for up to max_rows tokens: with room for one chunk's dZ and packed
// hidden states, for want_G chunks' (the size queries), or, given a workspace of ws_bytes, for as many
// chunks of both as fit, so that the two products run once per group of G chunks.
static Layout layout(int64_t max_rows, int64_t V, int64_t D, size_t ws_bytes = 0, int64_t want_G = 0,
                     Room room = kAll) {
  const bool pack = room != kLeast;
  Layout L;
  L.pack = pack;
  L.Tc = std::max<int64_t>(1, std::min<int64_t>(max_rows, kChunk));
  const int64_t chunks = (std::max<int64_t>(max_rows, 1) + L.Tc - 1) / L.Tc;
  const int64_t n_nt = (V + BN - 1) / BN;
  L.n_nt = n_nt;
  L.vb = pack ? vb_tiles(L.Tc, n_nt) : kMaxVb;
  L.n_vb = (n_nt + L.vb - 1) / L.vb;
  L.n_part = kParts * ((n_nt + kMaxVb - 1) / kMaxVb);
  L.tile_parts = L.vb < kMaxVb;
  L.ldz = (V + 7) / 8 * 8;
  auto al = al256;
  size_t off = kWsHeader + al(static_cast<size_t>(std::max<int64_t>(max_rows, 0)) * sizeof(double));
  L.off_partials = off;
  off += partials_bytes(L);
  if (!pack) off += al(static_cast<size_t>(L.Tc) * 32);  // unused: what was too small for a call stays too small
  L.off_tmax = off;
  off += al(static_cast<size_t>(L.Tc * n_nt) * sizeof(float));
  L.off_idx = off;  // the number of trained tokens (64 words apart from the list), then the list
  if (pack) off += 256 + al(static_cast<size_t>(std::max<int64_t>(max_rows, 1)) * sizeof(int32_t));
  L.off_counts = off;
  if (pack && select_blocks(max_rows) > kSelAlone) off += al(static_cast<size_t>(select_blocks(max_rows)) * sizeof(int32_t));
  L.parts = room == kAll && max_rows <= kChunk ? dh_parts(L.Tc, V, D) : 1;
  L.off_parts = off;
  if (L.parts > 1) off += al(static_cast<size_t>(L.parts * L.Tc * D) * sizeof(float));
  // the group's chunks: the logits gradient and the packed hidden states of each
  const size_t chunk_dz = static_cast<size_t>(L.Tc * L.ldz) * 2;
  const size_t chunk_h = pack ? al(static_cast<size_t>(L.Tc * D) * 2) : 0;
  int64_t G = want_G;
  if (ws_bytes > off) G = static_cast<int64_t>((ws_bytes - off) / (chunk_dz + chunk_h));
  L.G = std::max<int64_t>(1, std::min<int64_t>(G, chunks));
  L.off_h = off;
  off += static_cast<size_t>(L.G) * chunk_h;
  L.off_dz = off;
  off += al(static_cast<size_t>(L.G) * chunk_dz);
  L.total = off;
  return L;
}

// The layout that a workspace of ws_bytes gives (Layout::total above ws_bytes: too small). The
// size that rl_workspace_size gives for these T, V and D has room for everything; one made for
// other sizes may not.
static Layout layout_in(int64_t T, int64_t V, int64_t D, size_t ws_bytes) {
  for (Room room : {kAll, kPacked}) {
    const Layout L = layout(T, V, D, ws_bytes, 0, room);
    if (L.total <= ws_bytes) return L;
  }
  return layout(T, V, D, ws_bytes, 0, kLeast);
}

// Which passes use the 256 x 512 form: bit 0 the forward-only statistics (STATS), bit 1 the
// loss call's statistics pass (STATS_P). Measured at 32,768 x 4,096 x 151,936 (back to back,
// same box): the forward-only call 24.24-24.36 ms wide (one epilogue group; 23.54-23.65 ms with
// two) against 24.81 ms with 256 x 256 tiles; the loss call 70.9-71.9 ms with wide statistics
// tiles (two epilogue groups) against 69.7-70.1 ms with 256 x 256 ones: its heavier epilogue,
// which stores the exponentials, is hidden behind the MMAs only with two accumulators.
#ifndef RL_HEAD_WIDE
#define RL_HEAD_WIDE 1
#endif

template <int MODE, bool TILE_PARTS>
static rl_status launch_head_form(const CUtensorMap& mh, const CUtensorMap& mw, const HeadArgs& a, cudaStream_t s) {
  constexpr bool kWide = ((RL_HEAD_WIDE >> MODE) & 1) != 0;
  auto kern = [] {
    if constexpr (kWide) return head_wide_kernel<MODE, TILE_PARTS>;
    else return head_kernel<MODE, kPair, TILE_PARTS>;
  }();
  constexpr size_t smem = kWide ? kSmemW : (kPair ? kSmem2 : kSmem);
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return cuda_error(e, "cudaDeviceGetAttribute");
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.blockDim = dim3(kWide ? kThreadsW : kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  static std::mutex mu;
  static std::map<std::pair<int, int>, int> resident;  // pairs resident at once (pair form)
  int max_pairs = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto key = std::make_pair(dev, MODE);
    auto it = resident.find(key);
    if (it == resident.end()) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
      if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(head_kernel)");
      int n = sms;
      if constexpr (kPair || kWide) {
        cfg.gridDim = dim3(2);
        e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
        if (e != cudaSuccess) return cuda_error(e, "cudaOccupancyMaxActiveClusters(head_kernel)");
        if (n <= 0) return set_error(RL_ERR_UNSUPPORTED, "head_kernel: no CTA pair fits on the device");
      }
      it = resident.emplace(key, n).first;
    }
    max_pairs = it->second;
  }
  if constexpr (kPair || kWide) {
    // persistent: one 2-CTA cluster per resident pair, work items of 256 tokens x one vocabulary block
    const int items = static_cast<int>((std::min<int64_t>(a.tok.Tc, a.tok.T) + 2 * BM - 1) / (2 * BM)) * a.n_vb;
    const int pairs = std::max(1, std::min(items, max_pairs));
    cfg.gridDim = dim3(2 * pairs);
    e = cudaLaunchKernelEx(&cfg, kern, mh, mw, a);
    if (e != cudaSuccess) return cuda_error(e, "cudaLaunchKernelEx(head_kernel)");
  } else {
    const int items = static_cast<int>((std::min<int64_t>(a.tok.Tc, a.tok.T) + BM - 1) / BM) * a.n_vb;
    kern<<<std::min(items, sms), kThreads, smem, s>>>(mh, mw, a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "head_kernel launch");
  }
  return RL_OK;
}

template <int MODE>
static rl_status launch_head(const CUtensorMap& mh, const CUtensorMap& mw, const HeadArgs& a, bool tile_parts,
                             cudaStream_t s) {
  return tile_parts ? launch_head_form<MODE, true>(mh, mw, a, s) : launch_head_form<MODE, false>(mh, mw, a, s);
}

}  // namespace head

size_t head_workspace_bytes(int64_t max_rows, int64_t V, int64_t D) {
  return head::layout(max_rows, V, D).total;
}

size_t head_workspace_bytes_grouped(int64_t max_rows, int64_t V, int64_t D, int64_t group_tokens) {
  const int64_t g = (std::max<int64_t>(group_tokens, 1) + head::kChunk - 1) / head::kChunk;
  return head::layout(max_rows, V, D, 0, g).total;
}

// The forward-only call needs the status word and one chunk's partials, which sit at the
// same offset as in the loss layout's header; rl_workspace_size(T, V, D) always suffices.
// It keeps the loss call's chunk of 4,096 tokens: the chunk's hidden states (32 MB at
// D = 4,096) and the W tiles in use then stay in L2 together. Measured at 32,768 x 4,096 x
// 151,936: chunks of 4,096 tokens give 24.8 ms per forward-only call (70.9 ms per loss call),
// 3,072 and 6,144 are within 2%, 8,192 takes 26.7 ms (73.1), and 32,768 takes 31.5 ms: the
// hidden states (256 MB) then evict W's tiles from the 129 MB L2.
static size_t head_logp_workspace_bytes(const head::Layout& L) {
  return kWsHeader + head::partials_bytes(L);
}

}  // namespace rl

extern "C" rl_status rl_fused_head_loss_fwd_bwd(
    const void* hidden, const void* weight, int64_t T, int64_t D, int64_t V, const int32_t* token_ids,
    const uint8_t* mask, const int32_t* token_traj, int32_t n_traj, const float* adv, const float* coef,
    const float* old_logp, const float* ref_logp, const float* rollout_logp, const rl_loss_params* params,
    void* d_hidden, rl_dtype d_hidden_dtype, float* d_weight, double* loss_accum, float* token_stats, void* ws,
    size_t ws_bytes, rl_stream_t stream) {
  using namespace rl;
  using namespace rl::head;
  clear_error();
  if (T < 0 || D < 64 || V < 1 || n_traj < 0)
    return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_loss_fwd_bwd: need T >= 0, D >= 64, V >= 1, n_traj >= 0");
  if (D % 64 != 0) return set_error(RL_ERR_UNSUPPORTED, "rl_fused_head_loss_fwd_bwd: D must be a multiple of 64");
  if (T > INT32_MAX || V > static_cast<int64_t>(kMaxTilesSmem) * BN || D > 65536)
    return set_error(RL_ERR_UNSUPPORTED, "rl_fused_head_loss_fwd_bwd: T above 2^31 - 1, V above 524,288 or D above 65536");
  if (!params || !loss_accum || !ws) return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_loss_fwd_bwd: NULL argument");
  if (d_hidden_dtype != RL_BF16 && d_hidden_dtype != RL_F32)
    return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_loss_fwd_bwd: unknown d_hidden dtype");
  if (params->kl_estimator != 0 && params->kl_estimator != 3)
    return set_error(RL_ERR_UNSUPPORTED, "rl_fused_head_loss_fwd_bwd: kl_estimator must be 0 or 3");
  if (params->token_level_adv != 0 && params->token_level_adv != 1)
    return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_loss_fwd_bwd: token_level_adv must be 0 or 1");
  const Layout L = layout_in(T, V, D, ws_bytes);
  if (ws_bytes < L.total)
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL,
                     "rl_fused_head_loss_fwd_bwd: workspace smaller than rl_workspace_size(T, V, D)");
  if (T == 0) return RL_OK;
  if (!hidden || !weight || !token_ids || !mask || !token_traj || !old_logp || !d_hidden || !d_weight ||
      (n_traj > 0 && (!adv || !coef)) || (params->token_level_adv && !adv))
    return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_loss_fwd_bwd: NULL array argument");
  if (!aligned16(hidden) || !aligned16(weight) || !aligned16(d_hidden) || !aligned16(d_weight) || !aligned16(ws))
    return set_error(RL_ERR_ALIGNMENT,
                     "rl_fused_head_loss_fwd_bwd: hidden, weight, d_hidden, d_weight and ws must be 16-byte aligned");

  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  char* wsb = static_cast<char*>(ws);
  int32_t* status = reinterpret_cast<int32_t*>(wsb);
  double* row_loss = reinterpret_cast<double*>(wsb + ws_row_loss_offset());
  float4* partials = reinterpret_cast<float4*>(wsb + L.off_partials);
  float* tmax = reinterpret_cast<float*>(wsb + L.off_tmax);
  uint16_t* dz_base = reinterpret_cast<uint16_t*>(wsb + L.off_dz);
  rl_status st = RL_OK;
  const bool kl_on = params->kl_estimator == 3 && params->kl_coef != 0.f && ref_logp != nullptr;
  const bool ent = params->entropy_coef != 0.f || token_stats != nullptr;

  CUtensorMap mw;
  st = make_map(&mw, weight, D, V, kWBoxRows);
  if (st != RL_OK) return st;
  const int n_nt = static_cast<int>(L.n_nt);
  const int64_t group_rows = L.G * L.Tc;
  Tokens tok = {};
  tok.T = static_cast<int32_t>(T);
  tok.Tc = static_cast<int32_t>(L.Tc);
  tok.G = static_cast<int32_t>(L.G);
  uint16_t* packed = reinterpret_cast<uint16_t*>(wsb + L.off_h);
  cudaError_t e = cudaSuccess;
  if (L.pack) {
    SelectArgs sa = {};
    sa.T = tok.T;
    sa.V = static_cast<int>(V);
    sa.n_traj = n_traj;
    sa.token_ids = token_ids;
    sa.mask = mask;
    sa.token_traj = token_traj;
    sa.coef = coef;
    sa.n_dev = reinterpret_cast<int32_t*>(wsb + L.off_idx);
    sa.idx = reinterpret_cast<int32_t*>(wsb + L.off_idx + 256);
    sa.row_loss = row_loss;
    sa.token_stats = token_stats;
    sa.status = status;
    const unsigned blocks = static_cast<unsigned>(select_blocks(T));
    if (blocks > kSelAlone) {
      sa.counts = reinterpret_cast<int32_t*>(wsb + L.off_counts);
      head_count_kernel<<<blocks, kSelThreads, 0, s>>>(sa);
      e = cudaGetLastError();
      if (e != cudaSuccess) return cuda_error(e, "head_count_kernel launch");
    }
    head_select_kernel<<<blocks, kSelThreads, 0, s>>>(sa);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "head_select_kernel launch");
    tok.idx = sa.idx;
    tok.n_dev = sa.n_dev;
  }
  // as many chunks as the tokens could need (the trained ones may need fewer: the kernels of a
  // chunk without tokens return at once)
  const int n_chunks = static_cast<int>((T + L.Tc - 1) / L.Tc);
  for (int c = 0; c < n_chunks; ++c) {
    const int64_t g0 = c / L.G * group_rows;  // first token of this chunk's group
    const int64_t gn = std::min<int64_t>(group_rows, T - g0);
    const uint16_t* h_group = L.pack ? packed : static_cast<const uint16_t*>(hidden) + g0 * D;
    const int64_t h_rows = L.pack ? group_rows : gn;
    const int Tc = static_cast<int>(std::min<int64_t>(L.Tc, T));
    if (L.pack) {
      GatherArgs ga = {};
      ga.tok = tok;
      ga.chunk = c;
      ga.D = static_cast<int>(D);
      ga.dh_bytes = d_hidden_dtype == RL_BF16 ? 2 : 4;
      ga.hidden = static_cast<const uint16_t*>(hidden);
      ga.packed = packed;
      ga.d_hidden = static_cast<char*>(d_hidden);
      head_gather_kernel<<<std::min((Tc + 7) / 8, 152 * 8), 256, 0, s>>>(ga);
      e = cudaGetLastError();
      if (e != cudaSuccess) return cuda_error(e, "head_gather_kernel launch");
    }
    CUtensorMap mh;
    st = make_map(&mh, h_group, D, h_rows, BM);
    if (st != RL_OK) return st;
    HeadArgs ha = {};
    ha.tok = tok;
    ha.chunk = c;
    ha.D = static_cast<int>(D);
    ha.V = static_cast<int>(V);
    ha.n_nt = n_nt;
    ha.vb_tiles = static_cast<int>(L.vb);
    ha.n_vb = static_cast<int>(L.n_vb);
    ha.ent = ent ? 1 : 0;
    ha.token_ids = token_ids;
    ha.partials = partials;
    ha.dz = dz_base;
    ha.ldz = L.ldz;
    ha.tmax = tmax;
    ha.status = status;
    st = launch_head<STATS_P>(mh, mw, ha, L.tile_parts, s);
    if (st != RL_OK) return st;

    DzArgs da = {};
    da.tok = tok;
    da.chunk = c;
    da.V = static_cast<int>(V);
    da.n_nt = n_nt;
    da.n_part = static_cast<int>(L.n_part);
    da.n_tile = L.tile_parts ? n_nt : 0;
    da.n_traj = n_traj;
    da.split = dz_split(Tc, V);
    da.ent = params->entropy_coef != 0.f ? 1 : 0;
    da.partials = partials;
    da.tmax = tmax;
    da.dz = dz_base;
    da.ldz = L.ldz;
    da.token_ids = token_ids;
    da.mask = mask;
    da.token_traj = token_traj;
    da.adv = adv;
    da.coef = coef;
    da.old_logp = old_logp;
    da.ref_logp = kl_on ? ref_logp : nullptr;
    da.rollout_logp = rollout_logp;
    da.clip_lo = 1.f - params->clip_eps_low;
    da.clip_hi = 1.f + params->clip_eps_high;
    da.beta = kl_on ? params->kl_coef : 0.f;
    da.alpha = params->entropy_coef;
    da.tis_cap = rollout_logp ? params->tis_cap : 0.f;
    da.adv_per_row = params->token_level_adv;
    da.row_loss = row_loss;
    da.counter = reinterpret_cast<uint32_t*>(wsb + kWsHeadCounterOffset);
    da.token_stats = token_stats;
    da.status = status;
    head_dz_kernel<<<std::min(Tc * da.split, 152 * 16), kDzThreads, 0, s>>>(da);
    e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "head_dz_kernel launch");

    // after the group's last chunk, the two products over the group's tokens
    if ((c + 1) % L.G == 0 || c + 1 == n_chunks) {
      float* parts = L.parts > 1 ? reinterpret_cast<float*>(wsb + L.off_parts) : nullptr;
      st = head_grad(tok, static_cast<int>(c / L.G), h_rows, dz_base, L.ldz, V, weight, h_group, D, d_hidden,
                     d_hidden_dtype, d_weight, parts, static_cast<int>(L.parts), row_loss,
                     c + 1 == n_chunks ? loss_accum : nullptr,
                     reinterpret_cast<uint32_t*>(wsb + kWsHeadCounterOffset), status, s);
      if (st != RL_OK) return st;
    }
  }
  return RL_OK;
}

extern "C" rl_status rl_fused_head_token_logprobs(const void* hidden, const void* weight, int64_t T, int64_t D,
                                                  int64_t V, const int32_t* token_ids, float* logp_out,
                                                  float* entropy_out, float* lse_out, void* ws, size_t ws_bytes,
                                                  rl_stream_t stream) {
  using namespace rl;
  using namespace rl::head;
  clear_error();
  if (T < 0 || D < 64 || V < 1)
    return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_token_logprobs: need T >= 0, D >= 64, V >= 1");
  if (D % 64 != 0) return set_error(RL_ERR_UNSUPPORTED, "rl_fused_head_token_logprobs: D must be a multiple of 64");
  if (T > INT32_MAX || V > INT32_MAX || D > 65536)
    return set_error(RL_ERR_UNSUPPORTED, "rl_fused_head_token_logprobs: T or V above 2^31 - 1, or D above 65536");
  if (!ws) return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_token_logprobs: NULL workspace");
  // the smaller work items where the tiles' partials fit, else blocks of 16 tiles
  Layout L = layout(T, V, D);
  if (ws_bytes < head_logp_workspace_bytes(L)) L = layout(T, V, D, 0, 0, kLeast);
  if (ws_bytes < head_logp_workspace_bytes(L))
    return set_error(RL_ERR_WORKSPACE_TOO_SMALL, "rl_fused_head_token_logprobs: workspace too small");
  if (T == 0) return RL_OK;
  if (!hidden || !weight || !token_ids || !logp_out)
    return set_error(RL_ERR_INVALID_ARG, "rl_fused_head_token_logprobs: NULL array argument");
  if (!aligned16(hidden) || !aligned16(weight) || !aligned16(ws))
    return set_error(RL_ERR_ALIGNMENT, "rl_fused_head_token_logprobs: hidden, weight and ws must be 16-byte aligned");

  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  char* wsb = static_cast<char*>(ws);
  int32_t* status = reinterpret_cast<int32_t*>(wsb);
  float4* partials = reinterpret_cast<float4*>(wsb + kWsHeader);
  CUtensorMap mw;
  rl_status st = make_map(&mw, weight, D, V, kWBoxRows);
  if (st != RL_OK) return st;
  Tokens tok = {};
  tok.T = static_cast<int32_t>(T);
  tok.Tc = static_cast<int32_t>(L.Tc);
  tok.G = 1;
  for (int c = 0; c * L.Tc < T; ++c) {
    const int64_t t0 = c * L.Tc;
    const int Tc = static_cast<int>(std::min<int64_t>(L.Tc, T - t0));
    CUtensorMap mh;
    st = make_map(&mh, static_cast<const uint16_t*>(hidden) + t0 * D, D, Tc, BM);
    if (st != RL_OK) return st;
    HeadArgs ha = {};
    ha.tok = tok;
    ha.chunk = c;
    ha.D = static_cast<int>(D);
    ha.V = static_cast<int>(V);
    ha.n_nt = static_cast<int>(L.n_nt);
    ha.vb_tiles = static_cast<int>(L.vb);
    ha.n_vb = static_cast<int>(L.n_vb);
    ha.ent = entropy_out ? 1 : 0;
    ha.token_ids = token_ids;
    ha.partials = partials;
    ha.status = status;
    st = launch_head<STATS>(mh, mw, ha, L.tile_parts, s);
    if (st != RL_OK) return st;
    LogpMergeArgs ma = {};
    ma.tok = tok;
    ma.chunk = c;
    ma.V = static_cast<int>(V);
    ma.n_part = static_cast<int>(L.n_part);
    ma.n_tile = L.tile_parts ? ha.n_nt : 0;
    ma.partials = partials;
    ma.token_ids = token_ids;
    ma.logp_out = logp_out;
    ma.entropy_out = entropy_out;
    ma.lse_out = lse_out;
    ma.status = status;
    head_logp_merge_kernel<<<(Tc + kMergeRows - 1) / kMergeRows, kMergeThreads, 0, s>>>(ma);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_error(e, "head_logp_merge_kernel launch");
  }
  return RL_OK;
}
