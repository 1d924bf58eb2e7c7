// The fused head's tokens as its kernels see them: the whole call's, or the packed list of the
// trained ones (whose number only the device knows), cut into chunks and groups of chunks.
#pragma once

#include <cstdint>

#include "rl_device.cuh"

namespace rl {

struct Tokens {
  int32_t T, Tc;         // tokens of the call; most tokens of a chunk
  int32_t G;             // chunks per group
  const int32_t* idx;    // null: every token, in order; else the trained tokens' list
  const int32_t* n_dev;  // its length
};

struct Chunk {
  int64_t first;   // the chunk's first token: position in the list
  int32_t count;   // its tokens
  int32_t padded;  // rows up to which the packed buffers are filled (zeros past count)
  int32_t row;     // the chunk's first row in the group's buffers
};

constexpr int32_t kTokenBlock = 64;  // tokens per contraction block of the product over tokens

// Tokens per chunk: Tc, or, for the packed list, the list cut into as few chunks as Tc allows, of
// about the same size (whole 256-row tiles): 4,100 tokens are two chunks of 2,304 and 1,796, not
// 4,096 and 4.
__device__ __forceinline__ int32_t chunk_size(const Tokens& k, int32_t n) {
  if (!k.idx) return k.Tc;
  const int32_t nc = (n + k.Tc - 1) / k.Tc;
  if (nc <= 1) return k.Tc;
  const int32_t per = ((n + nc - 1) / nc + 255) / 256 * 256;
  return per < k.Tc ? per : k.Tc;
}

__device__ __forceinline__ Chunk chunk_of(const Tokens& k, int32_t c) {
  const int32_t n = k.n_dev ? *k.n_dev : k.T;
  const int32_t size = chunk_size(k, n);
  Chunk ch;
  ch.first = static_cast<int64_t>(c) * size;
  const int64_t left = n - ch.first;
  ch.count = static_cast<int32_t>(left < 0 ? 0 : left < size ? left : size);
  ch.row = (c % k.G) * size;
  const int32_t up = (ch.count + kTokenBlock - 1) / kTokenBlock * kTokenBlock;
  ch.padded = k.idx ? (up < k.Tc ? up : k.Tc) : ch.count;
  return ch;
}

// The tokens of group g (its chunks lie one after another): first, count and row = 0.
__device__ __forceinline__ Chunk group_of(const Tokens& k, int32_t g) {
  const int32_t n = k.n_dev ? *k.n_dev : k.T;
  const int64_t size = static_cast<int64_t>(chunk_size(k, n)) * k.G;
  Chunk ch;
  ch.first = g * size;
  const int64_t left = n - ch.first;
  ch.count = static_cast<int32_t>(left < 0 ? 0 : left < size ? left : size);
  ch.padded = ch.count;
  ch.row = 0;
  return ch;
}

// Token of the chunk's (or group's) row r.
__device__ __forceinline__ int32_t token_of(const Tokens& k, const Chunk& ch, int64_t r) {
  return k.idx ? k.idx[ch.first + r] : static_cast<int32_t>(ch.first + r);
}

}  // namespace rl
