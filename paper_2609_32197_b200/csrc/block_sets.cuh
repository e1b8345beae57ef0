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

// words[kMaxWords]: the blocks of rank r.  The caller synchronises the block afterwards.
__device__ __forceinline__ void rank_words(const int32_t* __restrict__ rank, int NB, int r, uint32_t* words) {
  if (threadIdx.x < kMaxWords) words[threadIdx.x] = 0u;
  __syncthreads();
  for (int j = threadIdx.x; j < NB; j += blockDim.x)
    if (rank[j] == r) atomicOr(&words[j >> 5], 1u << (j & 31));
}

// list[]: the blocks of the set in ascending order; returns their number.  Synchronises before and after.
__device__ __forceinline__ int list_blocks(const uint32_t* words, int NB, uint16_t* list) {
  __syncthreads();
  int n = 0;
  for (int w = 0; w < (NB + 31) / 32; ++w) n += __popc(words[w]);
  for (int j = threadIdx.x; j < NB; j += blockDim.x) {
    const uint32_t word = words[j >> 5];
    if ((word >> (j & 31)) & 1u) {
      int pos = __popc(word & ((1u << (j & 31)) - 1u));
      for (int w = 0; w < (j >> 5); ++w) pos += __popc(words[w]);
      list[pos] = (uint16_t)j;
    }
  }
  __syncthreads();
  return n;
}

}  // namespace sparsp
