// Step 1: mean-pool Q and K per block, score pooled-Q x pooled-K^T per head (fp32 SIMT GEMM with a
// fixed accumulation order), warp-level top-k per row.
//
// Arithmetic contract (the result decides which blocks are kept, so it is fixed to the operation):
//   pool : fp32 sum of the block's valid tokens in ascending token order starting from 0, then one
//          IEEE division by the valid count;
//   score: acc = fmaf(q_c, k_c, acc) from acc = 0, channel c ascending;
//   top-k: score descending, index ascending on equal scores, -0 == +0.
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace sparsp {

// ------------------------------------------------------------------------------------------------
// pool: a warp per (tensor, batch*head, block) tile, a CTA of its own.  The tile comes into shared memory as one TMA
// load (any token stride; rows behind the last token arrive as zeros), so all of it is in flight at once and as many
// tiles per multiprocessor as fit there; a lane then adds its 2 or 4 channels row by row, every channel one sequential
// chain.  HBM-bound where there are many tiles, one memory latency and the chain of `block` additions where there are
// few.  us of a whole mask call with loads through registers (8 to 32 rows in flight a lane) / this way: 40 heads x
// 75600 x 128 486 / 419, 24 x 24576 115 / 100 (pool alone 53.6 -> about 46, 6.5 TB/s), 48 x 17776 x 64 89 / 81, 2 x 13
// x 6034 x 64 token-major 18.6 / 13.1, 48 heads x 1558 token-major 23.9 / 14.5, 2 x 4096 x 64 11.7 / 9.9.
// ------------------------------------------------------------------------------------------------
template <int D>
__global__ void __launch_bounds__(32) pool_kernel(const __grid_constant__ CUtensorMap tmQ,
                                                  const __grid_constant__ CUtensorMap tmK, float* __restrict__ pq,
                                                  float* __restrict__ pk, int H, int NB, int b, int64_t N, int n_tiles,
                                                  int32_t* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ uint64_t full;
  __shared__ int s_abort;
  const int lane = threadIdx.x;
  const bool is_k = blockIdx.x >= (unsigned)n_tiles;
  const int t = is_k ? (int)blockIdx.x - n_tiles : (int)blockIdx.x;  // (batch*H + head) * NB + block
  const int bh = t / NB, blk = t - bh * NB;
  if (lane == 0) {
    s_abort = 0;
    ptx::mbar_init(&full, 1);
    ptx::mbar_init_fence();
  }
  enter_grid();
  if (lane == 0) {
    ptx::mbar_expect_tx(&full, (uint32_t)(b * D * 2));
    ptx::tma_load_4d(smem_raw, is_k ? &tmK : &tmQ, &full, 0, blk * b, bh % H, bh / H);
  }
  __syncwarp();
  ptx::mbar_wait_bounded(&full, 0, &s_abort, status, 50, 200000000LL);
  constexpr int W = D / 64;  // 32-bit words per lane and row
  const uint32_t* row = reinterpret_cast<const uint32_t*>(smem_raw) + lane * W;
  float acc[2 * W];
#pragma unroll
  for (int c = 0; c < 2 * W; ++c) acc[c] = 0.0f;
  // (a row behind the last token adds +0, which changes no sum: a sum that starts at +0 is never -0)
#pragma unroll 16
  for (int r = 0; r < b; ++r, row += D / 2) {
    uint32_t v[W];
    if (W == 2) {
      const uint2 x = *reinterpret_cast<const uint2*>(row);
      v[0] = x.x;
      v[W - 1] = x.y;
    } else {
      v[0] = *row;
    }
#pragma unroll
    for (int w = 0; w < W; ++w) {
      acc[2 * w] = __fadd_rn(acc[2 * w], __uint_as_float(v[w] << 16));
      acc[2 * w + 1] = __fadd_rn(acc[2 * w + 1], __uint_as_float(v[w] & 0xffff0000u));
    }
  }
  const float cntf = (float)min((int64_t)b, N - (int64_t)blk * b);
  float* dst = (is_k ? pk : pq) + (int64_t)t * D + lane * 2 * W;
#pragma unroll
  for (int w = 0; w < W; ++w)
    *reinterpret_cast<float2*>(dst + 2 * w) = make_float2(__fdiv_rn(acc[2 * w], cntf), __fdiv_rn(acc[2 * w + 1], cntf));
}

int launch_pool(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, float* pq, float* pk, char* ws,
                const WsLayout& L, cudaStream_t st) {
  CUtensorMap tq, tk;
  int rc;
  if ((rc = make_tile_tmap(&tq, Q, s, g, g.b, false)) != SPARSP_OK) return rc;
  if ((rc = make_tile_tmap(&tk, K, s, g, g.b, false)) != SPARSP_OK) return rc;
  const int n_tiles = g.B * g.H * g.NB;
  auto kern = g.d == 64 ? pool_kernel<64> : pool_kernel<128>;
  SPARSP_CUDA_OK(launch_kernel(kern, 2u * (unsigned)n_tiles, 32, (size_t)g.b * g.d * 2, st, tq, tk, pq, pk, g.H, g.NB, g.b,
                               g.N, n_tiles, (int32_t*)(ws + L.status)));
  return SPARSP_OK;
}

// ------------------------------------------------------------------------------------------------
// score: S[bh][i][j] = sum_c pQ[i][c] * pK[j][c] as one fused-multiply-add chain per output, c
// ascending (a no-split-K SIMT GEMM).  A CTA computes a 64 x 64 tile; a thread owns 4 rows x 4
// columns (columns tx, tx+16, tx+32, tx+48 so that its 16-byte shared-memory reads of pooled K never
// conflict), i.e. 16 independent chains fed by 8 vector loads per 4 channels.  Scores go to a
// workspace buffer: at most 83 MB, written and read once, ~25 us of HBM time on the largest workload.
// ------------------------------------------------------------------------------------------------
constexpr int kScoreTile = 64;
constexpr int kScoreThreads = 256;

template <int D>
__global__ void __launch_bounds__(kScoreThreads) score_kernel(const float* __restrict__ pq,
                                                              const float* __restrict__ pk, int NB,
                                                              float* __restrict__ scores) {
  enter_grid(pq, pk);
  constexpr int LD = D + 4;  // row pitch in floats: 16 bytes of skew per row
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sQ = reinterpret_cast<float*>(smem_raw);  // [64][LD]
  float* sK = sQ + kScoreTile * LD;                // [64][LD]
  const int64_t bh = blockIdx.z;
  const int row0 = blockIdx.y * kScoreTile, col0 = blockIdx.x * kScoreTile;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;

  for (int idx = threadIdx.x; idx < kScoreTile * (D / 4); idx += kScoreThreads) {
    const int r = idx / (D / 4), c4 = idx % (D / 4);
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f), k = q;
    if (row0 + r < NB) q = __ldg(reinterpret_cast<const float4*>(pq + (bh * NB + row0 + r) * D) + c4);
    if (col0 + r < NB) k = __ldg(reinterpret_cast<const float4*>(pk + (bh * NB + col0 + r) * D) + c4);
    *reinterpret_cast<float4*>(sQ + r * LD + c4 * 4) = q;
    *reinterpret_cast<float4*>(sK + r * LD + c4 * 4) = k;
  }
  __syncthreads();

  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;

#pragma unroll 4
  for (int c = 0; c < D; c += 4) {
    float4 q[4], k[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const float4*>(sQ + (ty * 4 + i) * LD + c);
#pragma unroll
    for (int j = 0; j < 4; ++j) k[j] = *reinterpret_cast<const float4*>(sK + (tx + 16 * j) * LD + c);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float a = acc[i][j];
        a = __fmaf_rn(q[i].x, k[j].x, a);
        a = __fmaf_rn(q[i].y, k[j].y, a);
        a = __fmaf_rn(q[i].z, k[j].z, a);
        a = __fmaf_rn(q[i].w, k[j].w, a);
        acc[i][j] = a;
      }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = row0 + ty * 4 + i;
    if (r >= NB) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int cidx = col0 + tx + 16 * j;
      if (cidx < NB) scores[(bh * NB + r) * NB + cidx] = acc[i][j];
    }
  }
}

static cudaError_t launch_score(const Geometry& g, const float* pq, const float* pk, float* scores, cudaStream_t st) {
  const size_t smem = (size_t)2 * kScoreTile * (g.d + 4) * 4;
  const unsigned nt = (unsigned)((g.NB + kScoreTile - 1) / kScoreTile);
  auto kern = g.d == 64 ? score_kernel<64> : score_kernel<128>;
  const cudaError_t e = ensure_dynamic_smem((const void*)kern, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(kern, dim3(nt, nt, (unsigned)(g.B * g.H)), kScoreThreads, smem, st, pq, pk, g.NB, scores);
}

// ------------------------------------------------------------------------------------------------
// top-k: one warp per (batch, head, query block) row.  The row's scores become order-preserving
// uint32 keys in registers (lane l holds blocks l, l + 32, ...); the warp finds the k-th largest key by bisection
// between the row's smallest and largest key with compares and a warp sum per step, which ends as soon as a trial value
// has exactly k keys at or above it (well before the 32 steps that a search bit by bit always takes), breaks ties
// towards the lower index, forces the text blocks on, and emits the mask words and the ascending kept list by
// ballot-prefix compaction.  Bound by instruction issue, a compare and an add per key and step: instances for several
// row lengths. 24 x 384 rows of 384: 19 us, 40 x 591 of 591: 79 us, 24 x 929 of 929: 136 us (29, 152 and 194 us with 32
// steps of one bit each and instances of 4, 8, 16 and 32 words; bisection by the keys instead of the scores: 18, 71 and
// 212 us).  Four CTAs per SM although the instances of 24 and 32 words spill for it: pool, score and selection of 24 x
// 929 rows 273 us, 296 with three and 340 with two; of 40 x 700 rows 267, 284 and 285.
// ------------------------------------------------------------------------------------------------
constexpr int kTopkWarps = 8;

__device__ __forceinline__ uint32_t score_key(float s) {
  if (s == 0.0f) s = 0.0f;  // -0 -> +0 so that they compare equal
  const uint32_t u = __float_as_uint(s);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float key_score(uint32_t key) {
  return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
}

// A key in (lo, hi] for the next step of a search, lo < hi: the one of the middle of the two scores, which halves
// evenly spread scores where the middle of the keys halves their exponents; or the middle key where that is no such key
// (ends that are infinite, not numbers or neighbours) and in every third step, so that the search ends after at most 96
// steps.
__device__ __forceinline__ uint32_t middle(uint32_t lo, uint32_t hi, int step) {
  const uint32_t by_score = score_key(0.5f * key_score(lo) + 0.5f * key_score(hi));
  return by_score > lo && by_score <= hi && step % 3 != 2 ? by_score : lo + ((hi - lo) >> 1) + 1;
}

struct TopkParams {
  int NB, Wd, nb_cand, topk, kept_cap;
  uint32_t* mask;
  int32_t *kv_list, *kv_count;
};

// One warp, one row: score(t) is the score of block t * 32 + lane, asked for candidates only.
template <int WMAX, typename Score>
__device__ __forceinline__ void select_row(const TopkParams& p, int64_t row, Score score) {
  const int lane = threadIdx.x & 31, NB = p.NB, Wd = p.Wd, nb_cand = p.nb_cand, topk = p.topk, kept_cap = p.kept_cap;
  uint32_t* mask = p.mask;
  int32_t *kv_list = p.kv_list, *kv_count = p.kv_count;
  // a block that is not a candidate (text, padding) holds the key 0, which no trial threshold (>= 1) counts
  uint32_t key[WMAX];
#pragma unroll
  for (int t = 0; t < WMAX; ++t) key[t] = (t < Wd && t * 32 + lane < nb_cand) ? score_key(score(t)) : 0u;

  const uint32_t lt_mask = (1u << lane) - 1u;
  // T with |{ candidates : key >= T }| == topk, or else the topk-th largest key (ties)
  uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
  for (int t = 0; t < WMAX; ++t) {
    lo = min(lo, t * 32 + lane < nb_cand ? key[t] : 0xffffffffu);
    hi = max(hi, key[t]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);  // all candidates are >= lo, at least topk of them
  hi = __reduce_max_sync(0xffffffffu, hi);  // fewer than topk are > hi
  for (int step = 0; lo < hi && topk < nb_cand; ++step) {
    const uint32_t trial = middle(lo, hi, step);
    int c = 0;
#pragma unroll
    for (int t = 0; t < WMAX; ++t) c += key[t] >= trial ? 1 : 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if (c >= topk) lo = trial;
    else hi = trial - 1;
    if (c == topk) break;
  }
  const uint32_t T = lo;
  int gt = 0;
#pragma unroll
  for (int t = 0; t < WMAX; ++t) gt += key[t] > T ? 1 : 0;
  gt = __reduce_add_sync(0xffffffffu, gt);
  const int need_eq = topk - gt;  // ties at T taken in ascending index order
  int eq_seen = 0, out_pos = 0;
#pragma unroll
  for (int t = 0; t < WMAX; ++t) {
    if (t < Wd) {
      const int j = t * 32 + lane;
      const bool cand = j < nb_cand;
      const bool is_eq = cand && key[t] == T;
      const uint32_t eq_ballot = __ballot_sync(0xffffffffu, is_eq);
      const bool take_eq = is_eq && (eq_seen + __popc(eq_ballot & lt_mask) < need_eq);
      eq_seen += __popc(eq_ballot);
      const bool keep = (cand && key[t] > T) || take_eq || (j >= nb_cand && j < NB);
      const uint32_t word = __ballot_sync(0xffffffffu, keep);
      if (lane == 0) mask[row * Wd + t] = word;
      if (kv_list && keep) {
        const int pos = out_pos + __popc(word & lt_mask);
        if (pos < kept_cap) kv_list[row * kept_cap + pos] = j;
      }
      out_pos += __popc(word);
    }
  }
  if (kv_count && lane == 0) kv_count[row] = out_pos;
}

template <int WMAX, typename Params>
__device__ __forceinline__ void select_stored_row(const Params& p, const float* scores, int64_t n_rows) {
  const int64_t row = (int64_t)blockIdx.x * kTopkWarps + (threadIdx.x >> 5);  // (batch*H + head) * NB + i
  if (row >= n_rows) return;
  const float* srow = scores + row * p.NB + (threadIdx.x & 31);
  select_row<WMAX>(p, row, [&](int t) { return __ldcs(srow + t * 32); });
}

template <int WMAX>  // mask words per row this instance can hold (keys live in registers: WMAX per lane)
__global__ void __launch_bounds__(kTopkWarps * 32, WMAX <= 12 ? 6 : 4)
    topk_kernel(const float* __restrict__ scores, int64_t n_rows, const TopkParams p) {
  enter_grid(scores);
  select_stored_row<WMAX>(p, scores, n_rows);
}

// ------------------------------------------------------------------------------------------------
// CDF-threshold selection (Section 8.1): per row, softmax over the candidate scores, keep the smallest
// top set by score (whole groups of equal scores) whose mass reaches tau.  The mass is counted in integers, so
// that the kept set does not depend on the order of the additions:
//   x_j = (S_j - max S) * (scale * log2 e)  (fp32);  p_j = exp2c(x_j)  (fp32: clamp at -125, nearest-integer
//   split, degree-5 Horner polynomial with fused multiply-adds, integer part added into the exponent field);
//   w_j = floor(p_j * 2^26);  Z = sum w_j;  kept = { key >= T } for the largest T with
//   mass{ key >= T } >= ceil(tau * Z), the product taken once in fp64.
// One warp per row; T is found by bisection over the order-preserving key space, which is valid
// because the mass of { key >= t } never grows with t, until a
// single key is left between its ends: 24 x 384 rows of 384 in 24 us (37 us with 32 steps of one bit).
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ float exp2c(float x) {
  x = fmaxf(x, -125.0f);
  const float fi = rintf(x);
  const float f = x - fi;
  float p = 0.0013400432653725147f;
  p = fmaf(p, f, 0.009676037356257439f);
  p = fmaf(p, f, 0.05550327152013779f);
  p = fmaf(p, f, 0.2402210682630539f);
  p = fmaf(p, f, 0.6931471824645996f);
  p = fmaf(p, f, 1.0000001192092896f);
  return __int_as_float(__float_as_int(p) + (int)fi * (1 << 23));
}

// Sum over the warp of one 32-bit partial sum per lane (each < 2^32, the total needs up to 37 bits): the halves of
// the partial sums are added by the warp-reduction instruction and put together again.
__device__ __forceinline__ unsigned long long warp_sum(uint32_t v) {
  const uint32_t lo = __reduce_add_sync(0xffffffffu, v & 0xffffu), hi = __reduce_add_sync(0xffffffffu, v >> 16);
  return ((unsigned long long)hi << 16) + lo;
}

struct CdfParams {
  int NB, Wd, nb_cand;
  float tau, c;
  uint32_t* mask;
  int32_t* kv_count;
};

template <int WMAX, typename Score>
__device__ __forceinline__ void select_row(const CdfParams& p, int64_t row, Score score) {
  const int lane = threadIdx.x & 31, NB = p.NB, Wd = p.Wd, nb_cand = p.nb_cand;
  const float tau = p.tau, c = p.c;
  uint32_t* mask = p.mask;
  int32_t* kv_count = p.kv_count;
  // lane l holds blocks l, l + 32, ...  A block that is not a candidate holds key 0 (no trial threshold, all
  // >= 1, selects it) and the weight 0.
  uint32_t key[WMAX];
  uint32_t w[WMAX];
  float mx = -INFINITY;
#pragma unroll
  for (int t = 0; t < WMAX; ++t) {
    const int j = t * 32 + lane;
    const bool cand = t < Wd && j < nb_cand;
    const float s = cand ? score(t) : -INFINITY;
    w[t] = __float_as_uint(s);
    key[t] = cand ? score_key(s) : 0u;
    mx = fmaxf(mx, s);
  }
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
  uint32_t acc = 0;  // at most 32 terms of at most 2^26 + 8 each
#pragma unroll
  for (int t = 0; t < WMAX; ++t) {
    const int j = t * 32 + lane;
    uint32_t wj = 0u;
    if (t < Wd && j < nb_cand) {
      // the scaling is exact, the conversion truncates
      wj = __float2uint_rz(__fmul_rn(exp2c(__fmul_rn(__fsub_rn(__uint_as_float(w[t]), mx), c)), 67108864.0f));
      acc += wj;
    }
    w[t] = wj;
  }
  const unsigned long long theta = (unsigned long long)ceil(__dmul_rn((double)tau, (double)warp_sum(acc)));
  // a T with the same { key >= T } as the largest T with mass{ key >= T } >= theta: bisection between the row's
  // smallest and largest key, until a single key is left between the two ends
  uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
  for (int t = 0; t < WMAX; ++t) {
    lo = min(lo, t * 32 + lane < nb_cand ? key[t] : 0xffffffffu);
    hi = max(hi, key[t]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);  // mass{ key >= lo } >= theta
  hi = __reduce_max_sync(0xffffffffu, hi);  // mass{ key > hi } < theta
  int n_lo = nb_cand, n_hi = 0;             // keys >= lo, keys > hi
  for (int step = 0; lo < hi && n_lo - n_hi > 1; ++step) {
    const uint32_t trial = middle(lo, hi, step);
    uint32_t m = 0;
    int c = 0;
#pragma unroll
    for (int t = 0; t < WMAX; ++t) {
      m += key[t] >= trial ? w[t] : 0u;
      c += key[t] >= trial ? 1 : 0;
    }
    c = __reduce_add_sync(0xffffffffu, c);
    if (warp_sum(m) >= theta) {
      lo = trial;
      n_lo = c;
    } else {
      hi = trial - 1;
      n_hi = c;
    }
  }
  // (theta 0: all weights are zero, as with a NaN or infinite maximum; then no score reaches the threshold)
  const uint32_t T = theta != 0 ? lo : 0xffffffffu;
  int cnt = 0;
#pragma unroll
  for (int t = 0; t < WMAX; ++t) {
    if (t < Wd) {
      const int j = t * 32 + lane;
      const bool keep = (j < nb_cand && key[t] >= T) || (j >= nb_cand && j < NB);
      const uint32_t word = __ballot_sync(0xffffffffu, keep);
      if (lane == 0) mask[row * Wd + t] = word;
      cnt += __popc(word);
    }
  }
  if (kv_count && lane == 0) kv_count[row] = cnt;
}

template <int WMAX>  // mask words per row this instance can hold (keys and terms live in registers)
__global__ void __launch_bounds__(kTopkWarps * 32, WMAX <= 12 ? 4 : WMAX <= 20 ? 3 : 2)
    cdf_kernel(const float* __restrict__ scores, int64_t n_rows, const CdfParams p) {
  enter_grid(scores);
  select_stored_row<WMAX>(p, scores, n_rows);
}

// ------------------------------------------------------------------------------------------------
// Scores and selection of short rows (up to 128 blocks) in one launch: a CTA keeps the pooled K of its head in shared
// memory and takes a few rows of it, a warp each, whose scores never leave the registers they are selected from.  Same
// chains, same selection.  What bounds it is the latency of the launch, of bringing pooled K in (16 warps, more than
// have a row) and of one row: few rows a CTA while all CTAs run at once, more where pooled K would be read too often.
// us of a whole mask call, two launches / this way: 2 heads x 64 blocks of d = 64 9.7 / 7.6, 7 x 21 of d = 128 13.5 /
// 7.7, 2 x 68 15.2 / 9.6, 5 x 108 18.3 / 12.0, 26 x 48 of d = 64 13.2 / 10.6, 48 x 128 of d = 128 85 / 82.  (8 warps
// and rows whatever the size: 7.6, 7.6, 12.8, 15.1, 10.9, 84.  Rows of up to 256 blocks: 7 x 147 21.1 -> 18.5, but 2 x
// 200 14.2 -> 17.5 and 24 x 256 60 -> 79.)
// ------------------------------------------------------------------------------------------------
constexpr int kShortWords = 4;
constexpr int kShortWarps = 16;

template <int D, typename Params>
__global__ void __launch_bounds__(kShortWarps * 32)
    short_rows_kernel(const float* __restrict__ pq, const float* __restrict__ pk, int rows, const Params p) {
  enter_grid(pq, pk);
  constexpr int LD = D + 4;  // row pitch in floats: 16 bytes of skew per row
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sK = reinterpret_cast<float*>(smem_raw);  // [NB][LD]
  float* sQ = sK + p.NB * LD;                      // [rows][D]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, NB = p.NB;
  const int64_t row0 = (int64_t)blockIdx.y * NB;   // of my head
  const int first = blockIdx.x * rows, n_rows = min(rows, NB - first);
  const float4* k4 = reinterpret_cast<const float4*>(pk + row0 * D);
  const float4* q4 = reinterpret_cast<const float4*>(pq + (row0 + first) * D);
  for (int idx = threadIdx.x; idx < n_rows * (D / 4); idx += kShortWarps * 32)
    reinterpret_cast<float4*>(sQ)[idx] = __ldg(q4 + idx);
#pragma unroll 8
  for (int idx = threadIdx.x; idx < NB * (D / 4); idx += kShortWarps * 32)
    *reinterpret_cast<float4*>(sK + idx / (D / 4) * LD + idx % (D / 4) * 4) = __ldg(k4 + idx);
  __syncthreads();
  if (warp >= n_rows) return;
  float score[kShortWords];
#pragma unroll
  for (int t = 0; t < kShortWords; ++t) score[t] = 0.0f;
  const float* q = sQ + warp * D;
#pragma unroll 4
  for (int c = 0; c < D; c += 4) {
    const float4 qv = *reinterpret_cast<const float4*>(q + c);
#pragma unroll
    for (int t = 0; t < kShortWords; ++t) {
      if (t * 32 < NB) {  // (lanes behind the last block take its row)
        const float4 kv = *reinterpret_cast<const float4*>(sK + min(t * 32 + lane, NB - 1) * LD + c);
        score[t] = __fmaf_rn(qv.x, kv.x, score[t]);
        score[t] = __fmaf_rn(qv.y, kv.y, score[t]);
        score[t] = __fmaf_rn(qv.z, kv.z, score[t]);
        score[t] = __fmaf_rn(qv.w, kv.w, score[t]);
      }
    }
  }
  select_row<kShortWords>(p, row0 + first + warp, [&](int t) { return score[t]; });
}

template <typename Params>
static cudaError_t launch_short_rows(const Geometry& g, const float* pq, const float* pk, const Params& p,
                                     cudaStream_t st) {
  const int64_t BH = (int64_t)g.B * g.H;
  auto groups = [&](int rows) { return (g.NB + rows - 1) / rows; };
  const int rows = BH * groups(4) <= 148 ? 4 : BH * groups(8) <= 2 * 148 ? 8 : kShortWarps;
  const size_t smem = (size_t)(g.NB * (g.d + 4) + rows * g.d) * 4;
  auto kern = g.d == 64 ? short_rows_kernel<64, Params> : short_rows_kernel<128, Params>;
  const cudaError_t e = ensure_dynamic_smem((const void*)kern, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_kernel(kern, dim3((unsigned)groups(rows), (unsigned)BH), kShortWarps * 32, smem, st, pq, pk, rows, p);
}
static bool rows_are_short(const Geometry& g) { return g.Wd <= kShortWords && (int64_t)g.B * g.H <= 65535; }

int launch_score_cdf(const Geometry& g, const float* pq, const float* pk, float* scores, float tau, float scale,
                     uint32_t* mask, int32_t* kv_count, cudaStream_t st) {
  const float c = scale * 1.4426950408889634f;  // fp32 product, as in the definition above
  const CdfParams p = {g.NB, g.Wd, g.nb_cand, tau, c, mask, kv_count};
  if (rows_are_short(g)) {
    SPARSP_CUDA_OK(launch_short_rows(g, pq, pk, p, st));
    return SPARSP_OK;
  }
  SPARSP_CUDA_OK(launch_score(g, pq, pk, scores, st));
  const int64_t n_rows = (int64_t)g.B * g.H * g.NB;
  const unsigned grid = (unsigned)((n_rows + kTopkWarps - 1) / kTopkWarps);
  auto kern = g.Wd <= 4 ? cdf_kernel<4> : g.Wd <= 8 ? cdf_kernel<8> :
              g.Wd <= 12 ? cdf_kernel<12> : g.Wd <= 16 ? cdf_kernel<16> : g.Wd <= 20 ? cdf_kernel<20> :
              g.Wd <= 24 ? cdf_kernel<24> : cdf_kernel<32>;
  SPARSP_CUDA_OK(launch_kernel(kern, grid, kTopkWarps * 32, 0, st, scores, n_rows, p));
  return SPARSP_OK;
}

int launch_score_topk(const Geometry& g, const float* pq, const float* pk, float* scores, int topk,
                      uint32_t* mask, int32_t* kv_list, int32_t* kv_count, cudaStream_t st) {
  const TopkParams p = {g.NB, g.Wd, g.nb_cand, topk, topk + (g.NB - g.nb_cand), mask, kv_list, kv_count};
  if (rows_are_short(g)) {
    SPARSP_CUDA_OK(launch_short_rows(g, pq, pk, p, st));
    return SPARSP_OK;
  }
  SPARSP_CUDA_OK(launch_score(g, pq, pk, scores, st));
  const int64_t n_rows = (int64_t)g.B * g.H * g.NB;
  const unsigned grid = (unsigned)((n_rows + kTopkWarps - 1) / kTopkWarps);
  auto kern = g.Wd <= 4 ? topk_kernel<4> : g.Wd <= 8 ? topk_kernel<8> :
              g.Wd <= 12 ? topk_kernel<12> : g.Wd <= 16 ? topk_kernel<16> : g.Wd <= 20 ? topk_kernel<20> :
              g.Wd <= 24 ? topk_kernel<24> : topk_kernel<32>;
  SPARSP_CUDA_OK(launch_kernel(kern, grid, kTopkWarps * 32, 0, st, scores, n_rows, p));
  return SPARSP_OK;
}

}  // namespace sparsp
