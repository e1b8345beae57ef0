// Consumer-side helpers of the demand-routed exchange: the mask of one hop (consumer rank's query
// blocks x producer rank's KV blocks) and the log-sum-exp merge of per-hop partial attention results.
// Both are small element-wise kernels; the merge is HBM-bound (reads two outputs, writes one).
#include <algorithm>

#include "block_sets.cuh"
#include "common.cuh"

namespace sparsp {

// hop[b][h][i][w] = (rank[i] == consumer and head_begin <= h < head_end) ? mask[b][h][i][w] & own_producer[w] : 0.  A
// lane handles one word of kHopRows rows (rows of fewer than 32 words share a warp); the producer's ownership words and
// the consumer's rows are bits in shared memory, built once per CTA.  A mask is a few MB, so this is latency: 40 heads
// x 591 rows x 19 words in 5.0 us (11.3 us with a thread per word that walked 32 ranks for its ownership bits, 7.5 with
// a pass over the ranks for each of the two sets, 6.5 with eight rows a lane).
constexpr int kHopThreads = 256;
constexpr int kHopRows = 4;

__global__ void __launch_bounds__(kHopThreads) hop_mask_kernel(const uint32_t* __restrict__ mask,
                                                               const int32_t* __restrict__ rank, int H, int NB, int Wd,
                                                               int64_t n_rows, int consumer, int producer,
                                                               int head_begin, int head_end,
                                                               uint32_t* __restrict__ hop) {
  enter_grid(mask, rank);
  __shared__ uint32_t own_s[kMaxWords], row_s[kMaxWords];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  {
    constexpr int kLooks = kMaxWords / (kHopThreads / 32);  // words a warp looks at, all loads in flight
    int owner[kLooks];
#pragma unroll
    for (int t = 0; t < kLooks; ++t) {
      const int j = (warp + t * (kHopThreads / 32)) * 32 + lane;
      owner[t] = j < NB ? rank[j] : -1;
    }
#pragma unroll
    for (int t = 0; t < kLooks; ++t) {
      const uint32_t own = __ballot_sync(0xffffffffu, owner[t] == producer);
      const uint32_t row = __ballot_sync(0xffffffffu, owner[t] == consumer);
      if (lane == 0) {
        own_s[warp + t * (kHopThreads / 32)] = own;
        row_s[warp + t * (kHopThreads / 32)] = row;
      }
    }
  }
  __syncthreads();
  int width = 1;  // lanes per row: the next power of two
  while (width < Wd) width <<= 1;
  const int per_warp = 32 / width, w = lane & (width - 1), sub = lane / width;
  if (w >= Wd) return;
  const int64_t first = ((int64_t)blockIdx.x * (kHopThreads / 32) + warp) * kHopRows * per_warp + sub;
  uint32_t v[kHopRows];
#pragma unroll
  for (int k = 0; k < kHopRows; ++k) {
    const int64_t row = first + k * per_warp;
    v[k] = 0u;
    if (row < n_rows) {
      const int64_t bh = row / NB;
      const int i = (int)(row - bh * NB), h = (int)(bh % H);
      if (((row_s[i >> 5] >> (i & 31)) & 1u) && h >= head_begin && h < head_end) v[k] = mask[row * Wd + w];
    }
  }
#pragma unroll
  for (int k = 0; k < kHopRows; ++k) {
    const int64_t row = first + k * per_warp;
    if (row < n_rows) hop[row * Wd + w] = v[k] & own_s[w];
  }
}

// Log-sum-exp merge.  Unit of work: one (batch, head, token block).  Without `rank` a CTA each; with `rank` given only
// those of the blocks of `consumer` in heads [head_begin, head_end) (one chunk of one hop of one rank; every other row
// stays untouched), which each CTA lists from the rank table and then walks.  O_a, O_b, O: bf16 with the shape's
// strides; lse: fp32 [B][H][N].
// A thread handles 8 columns of a row, kMergeRows rows at a time with all their loads in flight: a block of 64 tokens
// has two rows for each thread at d = 64 (40 registers, 6 CTAs per SM), four or eight everywhere else (80 registers, 3
// CTAs).  HBM-bound, us as it is / with four rows and 4 CTAs per SM, of which 3 fit, whatever the shape / with a CTA
// per block and a row of loads in flight: 40 heads x 591 blocks of 128 x 128 as a whole 350 / 460 / 360, an eighth of
// its blocks 60 / 71 / 73; 24 x 384 of 64 x 128 75 / 91 / 75, a quarter of them 13 / 14 / 17; 48 x 279 of 64 x 64 62 /
// 97 / 65, an eighth 11 / 15 / 13.  (Listing 1024 blocks takes longer than the merge of few heads in L2: half of the
// blocks of 8 heads x 1024 of 64 x 64 22 / 34 / 18.)
// A consumer's blocks are walked from behind: the attention before the merge wrote the last ones last, and they are
// still in L2 (an attention of 40 heads x 75600 hop by hop 2539 us, 2515 this way).
// O may be O_a or O_b and lse may be lse_a or lse_b (no pointer is declared restrict): a thread reads the 16 bytes it
// later writes, and the D/8 threads of a row are consecutive lanes of one warp, all of which have read the row's
// log-sum-exp values before its first thread writes the merged one.
// A row to which the second part adds nothing (lse_b = -inf: no kept block in this hop) has nothing to do when it is
// merged in place.
constexpr int kMergeThreads = 256;
constexpr int merge_ctas_per_sm(int rows) { return rows == 2 ? 6 : 3; }

template <int D, int kMergeRows>
__global__ void __launch_bounds__(kMergeThreads, merge_ctas_per_sm(kMergeRows))
    attn_merge_kernel(const __nv_bfloat16* Oa, const float* la, const __nv_bfloat16* Ob, const float* lb,
                      __nv_bfloat16* O, float* lse, int B, int H, int NB, int64_t N, int b, int64_t sB, int64_t sH,
                      int64_t sT, const int32_t* __restrict__ rank, int consumer, int head_begin, int head_end) {
  enter_grid(rank);
  constexpr int VPR = D / 8;
  constexpr int kPass = kMergeThreads / VPR;  // rows per pass of the CTA
  __shared__ uint32_t words_s[kMaxWords];
  __shared__ uint16_t own_s[kMaxBlocks];
  int n_own = NB;
  if (rank != nullptr) {
    rank_words(rank, NB, consumer, words_s);
    n_own = list_blocks(words_s, NB, own_s);
  }
  const int heads = head_end - head_begin;
  const int64_t n_units = (int64_t)B * heads * n_own;
  const int col = threadIdx.x % VPR, r0 = threadIdx.x / VPR;
  const bool in_place = O == Oa && lse == la;
  for (int64_t v = blockIdx.x; v < n_units; v += gridDim.x) {
    const int64_t u = rank != nullptr ? n_units - 1 - v : v;
    const int64_t bhi = u / n_own;
    const int k = (int)(u - bhi * n_own);
    const int blk = rank != nullptr ? own_s[k] : k;
    const int batch = (int)(bhi / heads), head = head_begin + (int)(bhi - (int64_t)batch * heads);
    const int64_t tok0 = (int64_t)blk * b;
    const int n_rows = (int)min((int64_t)b, N - tok0);
    const int64_t lrow = ((int64_t)batch * H + head) * N + tok0;
    const int64_t orow = (int64_t)batch * sB + (int64_t)head * sH + tok0 * sT + col * 8;
    for (int base = 0; base < n_rows; base += kPass * kMergeRows) {
      float a[kMergeRows], c[kMergeRows];
      uint4 va[kMergeRows], vb[kMergeRows];
      bool live[kMergeRows];
#pragma unroll
      for (int t = 0; t < kMergeRows; ++t) {
        const int r = base + t * kPass + r0;
        live[t] = r < n_rows;
        a[t] = live[t] ? la[lrow + r] : 0.0f;
        c[t] = live[t] ? lb[lrow + r] : 0.0f;
      }
#pragma unroll
      for (int t = 0; t < kMergeRows; ++t) {
        const int64_t off = orow + (int64_t)(base + t * kPass + r0) * sT;
        if (in_place && c[t] == -INFINITY && a[t] > -INFINITY) live[t] = false;
        if (live[t]) {
          va[t] = *reinterpret_cast<const uint4*>(Oa + off);
          vb[t] = *reinterpret_cast<const uint4*>(Ob + off);
        }
      }
      __syncwarp();  // every lane of a row has its log-sum-exp values
#pragma unroll
      for (int t = 0; t < kMergeRows; ++t) {
        if (!live[t]) continue;
        const int r = base + t * kPass + r0;
        float wa = 0.0f, wb = 0.0f, out_lse = -INFINITY;
        const float m = fmaxf(a[t], c[t]);
        if (m > -INFINITY) {
          const float ea = __expf(a[t] - m), eb = __expf(c[t] - m);
          const float tot = ea + eb;
          wa = ea / tot;
          wb = eb / tot;
          out_lse = m + __logf(tot);
        }
        const uint32_t xa[4] = {va[t].x, va[t].y, va[t].z, va[t].w}, xb[4] = {vb[t].x, vb[t].y, vb[t].z, vb[t].w};
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float a0 = __uint_as_float(xa[e] << 16), a1 = __uint_as_float(xa[e] & 0xffff0000u);
          const float b0 = __uint_as_float(xb[e] << 16), b1 = __uint_as_float(xb[e] & 0xffff0000u);
          const __nv_bfloat162 h2 = __floats2bfloat162_rn(a0 * wa + b0 * wb, a1 * wa + b1 * wb);
          w[e] = *reinterpret_cast<const uint32_t*>(&h2);
        }
        *reinterpret_cast<uint4*>(O + orow + (int64_t)r * sT) = make_uint4(w[0], w[1], w[2], w[3]);
        if (col == 0) lse[lrow + r] = out_lse;
      }
      __syncwarp();
    }
  }
}

int launch_hop_mask(const Geometry& g, const uint32_t* mask, const int32_t* rank, int consumer, int producer,
                    int head_begin, int head_end, uint32_t* hop, cudaStream_t st) {
  const int64_t n_rows = (int64_t)g.B * g.H * g.NB;
  int width = 1;
  while (width < g.Wd) width <<= 1;
  const int per_cta = kHopThreads / width * kHopRows;
  SPARSP_CUDA_OK(launch_kernel(hop_mask_kernel, (unsigned)((n_rows + per_cta - 1) / per_cta), kHopThreads, 0, st, mask,
                               rank, g.H, g.NB, g.Wd, n_rows, consumer, producer, head_begin, head_end, hop));
  return SPARSP_OK;
}

int launch_attn_merge(const sparsp_shape& s, const Geometry& g, const void* Oa, const float* la, const void* Ob,
                      const float* lb, void* O, float* lse, const int32_t* rank, int consumer, int head_begin,
                      int head_end, cudaStream_t st) {
  if (head_end <= head_begin) return SPARSP_OK;
  int sms = 0;
  SPARSP_CUDA_OK(sm_count(&sms));
  const int rows = g.d == 64 && g.b == 64 ? 2 : 4;
  auto kern = g.d == 128 ? attn_merge_kernel<128, 4> : rows == 2 ? attn_merge_kernel<64, 2> : attn_merge_kernel<64, 4>;
  const int64_t units = (int64_t)g.B * (head_end - head_begin) * g.NB;
  // Walkers: as many CTAs as fit the chip (twice as many: half of the blocks of 8 heads x 1024 of 64 x 64 22.8 us for
  // 21.9); in the four-row form twice as many (an attention of 40 heads x 75600 hop by hop 3.00 ms, as many 3.07, four
  // times 3.045).
  const int64_t walkers = (rows == 2 ? 1LL : 2LL) * merge_ctas_per_sm(rows) * sms;
  const unsigned grid = (unsigned)(rank ? std::min(units, walkers) : units);
  SPARSP_CUDA_OK(launch_kernel(kern, grid, kMergeThreads, 0, st, (const __nv_bfloat16*)Oa, la, (const __nv_bfloat16*)Ob,
                               lb, (__nv_bfloat16*)O, lse, g.B, g.H, g.NB, g.N, g.b, s.stride_batch, s.stride_head,
                               s.stride_token, rank, consumer, head_begin, head_end));
  return SPARSP_OK;
}

}  // namespace sparsp
