// Host-side internals shared by the library's translation units.
#pragma once

#include <cstddef>
#include <cstdint>
#include <string>

#include <cuda_runtime.h>

#include "rl_loss.h"

namespace rl {

// Workspace layout (offsets in bytes from the caller's workspace pointer):
//   [0, 256)                 header: int32 device status word at offset 0
//   [256, 256 + 8 * rows)    double loss contributions: one per cluster of the logits-path
//                            loss kernel (its rows' c_i * l_t added in row order), one per
//                            row for the fused head and the value loss
constexpr size_t kWsHeader = 256;

inline size_t ws_row_loss_offset() { return kWsHeader; }
// Header word counting the loss kernel's finished clusters (zeroed by rl_workspace_init; the
// last cluster of each launch resets it).
constexpr size_t kWsDoneOffset = 16;
// The same for the value loss kernel's finished CTAs.
constexpr size_t kWsValueDoneOffset = 20;
// Work-item counter of the fused head's backward products (set back by the rescale before it).
constexpr size_t kWsHeadCounterOffset = 24;
// The statistics summary's finished clusters, and its clusters' totals (5 doubles each, to the
// header's end).
constexpr size_t kWsSummaryDoneOffset = 28;
constexpr size_t kWsSummaryOffset = 32;

rl_status set_error(rl_status st, const std::string& msg);
rl_status cuda_error(cudaError_t e, const char* what);
void clear_error();

// Smallest workspace of the fused LM head for up to max_rows tokens (rl_head.cu).
size_t head_workspace_bytes(int64_t max_rows, int64_t V, int64_t D);
// The same, keeping the dZ of up to group_tokens tokens (whole chunks) at once.
size_t head_workspace_bytes_grouped(int64_t max_rows, int64_t V, int64_t D, int64_t group_tokens);

struct Tokens;  // rl_head_tokens.cuh

// Backward products of the fused LM head on the tensor cores (rl_head_grad.cu), one launch over
// the n tokens of one group: d_hidden = dZ W (stored in the tokens' rows, bf16 or fp32) and
// d_weight[V x D] += dZ^T H[n x D] (fp32), with dz the bf16 gradient of the logits of the group's
// tokens ([rows x V] at most, rows ldz elements apart) and hidden their hidden states in the same
// order. parts > 1 cuts dH's contraction over V into that many items per tile, whose fp32 sums
// ([parts][Tc x D] at part_sums) a second launch adds. With loss_accum (the call's last launch) the
// tok.T loss contributions at row_loss are added to it, in a fixed order. counter: a workspace word
// for the work-item counter, zero before the launch (head_dz_kernel sets it back).
rl_status head_grad(const Tokens& tok, int group, int64_t rows, const uint16_t* dz, int64_t ldz, int64_t V,
                    const void* weight, const void* hidden, int64_t D, void* d_hidden, rl_dtype dh_dtype,
                    float* d_weight, float* part_sums, int parts, const double* row_loss, double* loss_accum,
                    uint32_t* counter, int32_t* status, cudaStream_t s);

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace rl
