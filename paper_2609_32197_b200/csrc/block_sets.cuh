// Sets of blocks as bit words in shared memory, built by one CTA from the rank table (at most kMaxBlocks blocks).
// Every function is called by all threads of the block.
#pragma once

#include "common.cuh"

namespace sparsp {

constexpr int kMaxWords = kMaxBlocks / 32;

// Number of set bits in the words of lower lanes; *total = set bits in all 32 lanes' words.
__device__ __forceinline__ int bits_below(uint32_t word, int lane, int* total) {
  const int mine = __popc(word);
  int incl = mine;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, s);
    if (lane >= s) incl += v;
  }
  *total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - mine;
}

// own[p][w]: bit j % 32 of word j / 32 set iff rank[j] == p; a rank outside [0, P) owns nothing.
// The caller synchronises the block afterwards.
__device__ __forceinline__ void own_words(const int32_t* __restrict__ rank, int NB, int Wd, int P, uint32_t* own) {
  for (int idx = threadIdx.x; idx < P * Wd; idx += blockDim.x) own[idx] = 0u;
  __syncthreads();
  for (int j = threadIdx.x; j < NB; j += blockDim.x) {
    const int r = rank[j];
    if ((unsigned)r < (unsigned)P) atomicOr(&own[r * Wd + (j >> 5)], 1u << (j & 31));
  }
}

// words[kMaxWords]: the blocks of rank r, a warp per word with its loads in flight.  The caller synchronises the block
// afterwards.
__device__ __forceinline__ void rank_words(const int32_t* __restrict__ rank, int NB, int r, uint32_t* words) {
  const int lane = threadIdx.x & 31, n = (NB + 31) >> 5;
  if (threadIdx.x >= n && threadIdx.x < kMaxWords) words[threadIdx.x] = 0u;
#pragma unroll 4
  for (int w = threadIdx.x >> 5; w < n; w += blockDim.x >> 5) {
    const int j = w * 32 + lane;
    const uint32_t word = __ballot_sync(0xffffffffu, (j < NB ? rank[j] : ~r) == r);
    if (lane == 0) words[w] = word;
  }
}

// list[]: the blocks of the set in ascending order; returns their number.  Synchronises before and after.
__device__ __forceinline__ int list_blocks(const uint32_t* words, int NB, uint16_t* list) {
  __shared__ int before_s[kMaxWords + 1];  // blocks of the set in lower words; all of them
  __syncthreads();
  if (threadIdx.x < kMaxWords) {
    int total;
    before_s[threadIdx.x] = bits_below(words[threadIdx.x], threadIdx.x, &total);
    if (threadIdx.x == 0) before_s[kMaxWords] = total;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < NB; j += blockDim.x) {
    const uint32_t word = words[j >> 5];
    if ((word >> (j & 31)) & 1u) list[before_s[j >> 5] + __popc(word & ((1u << (j & 31)) - 1u))] = (uint16_t)j;
  }
  __syncthreads();
  return before_s[kMaxWords];
}

}  // namespace sparsp
