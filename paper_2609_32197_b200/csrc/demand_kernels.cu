// Step 2: per-rank per-head unions of required KV blocks, demand counts, exchange volume,
// pack-order offsets, the destination table, and the gather of K/V tiles into per-consumer buffers.
// Everything before the gather is small integer work on bit words; the gather is the HBM-bound part.
#include <algorithm>
#include <climits>

#include "block_sets.cuh"
#include "common.cuh"
#include "sm100_ptx.cuh"

namespace sparsp {

// One CTA per (batch, head, rank r) computes
//   U[b][r][h][w] = OR over the query blocks i of rank r of M[b][h][i][w]
//   cnt[b][r][p][h] = popcount(U[b][r][h] & own[p]),  own[p] = the blocks of rank p
// and, with `received` given, received[b][r][h], the number of entries packed for consumer r in head h: what the plan's
// CTAs need of the consumers before theirs.
// It reads the rows of its own query blocks only, whole words per lane (a row of up to 32 words is one coalesced
// request, shorter rows share one), so a mask row is read once in all and B*H*P CTAs are in flight; the ownership
// words are rebuilt per CTA from the rank table.  Latency-bound: the mask is a few MB.  (One CTA per (batch, head) with
// shared-memory atomics for all ranks at once: 20.6 us on 24 heads x 929 blocks, 8 ranks, 24 CTAs on 148 SMs; this
// split 8 us.)  OR does not depend on the order, so the bits are well defined.  A rank value outside [0, P) is ignored.
// Where a lane has several rows one behind the other (kLong) the lists are made without atomics and eight rows are in
// flight, the last ones too: us a plan in a graph, atomics and four rows / this way, 24 x 929, 8 ranks 7.6 / 5.6, 40 x
// 591, 8 ranks 8.2 / 7.4, 48 x 1000, 3 ranks 8.3 / 7.1.  With few rows the instructions that takes are what bounds many
// CTAs: 16 x 500, 16 ranks 6.2 / 6.8, 2 x 32 x 246, 10 ranks 7.7 / 8.9, 2 x 48 x 512, 16 ranks 15.0 / 18.5.
constexpr int kUnionThreads = 512, kUnionWarps = kUnionThreads / 32;
constexpr int kLongRows = 4;  // rows a lane from which on

__host__ __device__ __forceinline__ int lanes_per_row(int Wd) {  // the next power of two
  int width = 1;
  while (width < Wd) width <<= 1;
  return width;
}
static bool rows_are_long(const Geometry& g, int P) {
  return (g.NB + P - 1) / P >= kLongRows * kUnionWarps * (32 / lanes_per_row(g.Wd));
}

// own[p][Wd] of all ranks and the list of rank r's rows; returns their number.  Called by all threads, own_s zeroed
// before.
__device__ __forceinline__ int list_rows(const int32_t* __restrict__ rank, int NB, int Wd, int P, int r,
                                         uint32_t* own_s, uint16_t* rows_s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kOwn = kMaxWords / kUnionWarps;  // words of blocks a warp looks at
  uint32_t mine[kOwn];                           // my rank's blocks of them
  int rk[kOwn];
#pragma unroll
  for (int t = 0; t < kOwn; ++t) {
    const int j = (warp + t * kUnionWarps) * 32 + lane;
    rk[t] = j < NB ? rank[j] : -1;
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < kOwn; ++t) {
    mine[t] = __ballot_sync(0xffffffffu, rk[t] == r);
    const uint32_t same = __match_any_sync(0xffffffffu, rk[t]);
    if ((unsigned)rk[t] < (unsigned)P && lane == __ffs(same) - 1) own_s[rk[t] * Wd + warp + t * kUnionWarps] = same;
  }
  __syncthreads();
  int n_rows;
  const int before = bits_below(lane < Wd ? own_s[r * Wd + lane] : 0u, lane, &n_rows);
#pragma unroll
  for (int t = 0; t < kOwn; ++t) {
    const int first = __shfl_sync(0xffffffffu, before, (warp + t * kUnionWarps) & 31);
    if ((mine[t] >> lane) & 1u)
      rows_s[first + __popc(mine[t] & ((1u << lane) - 1u))] = (uint16_t)((warp + t * kUnionWarps) * 32 + lane);
  }
  __syncthreads();
  return n_rows;
}

// OR of the listed rows of kHeads masks m[NB][Wd], `pitch` words apart, of which the first n_heads are there, a word
// per lane and mask.  Called by all lanes of a warp, which takes its share of the rows, kInFlight of every mask at a
// time.
template <int kHeads, int kInFlight>
__device__ __forceinline__ void or_rows(const uint32_t* __restrict__ m, int64_t pitch, int n_heads,
                                        const uint16_t* rows_s, int n_rows, int Wd, int width,
                                        uint32_t (&acc)[kHeads]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per_warp = 32 / width, w = lane & (width - 1), step = kUnionWarps * per_warp;
#pragma unroll
  for (int h = 0; h < kHeads; ++h) acc[h] = 0u;
  for (int k0 = warp * per_warp + lane / width; k0 < n_rows; k0 += kInFlight * step) {
    uint32_t v[kHeads][kInFlight];
#pragma unroll
    for (int u = 0; u < kInFlight; ++u) {
      const int k = k0 + u * step;
      const bool there = k < n_rows && w < Wd;
      const uint32_t* at = m + (there ? (int64_t)rows_s[k] * Wd + w : 0);
#pragma unroll
      for (int h = 0; h < kHeads; ++h) v[h][u] = there && h < n_heads ? at[h * pitch] : 0u;
    }
#pragma unroll
    for (int h = 0; h < kHeads; ++h)
#pragma unroll
      for (int u = 0; u < kInFlight; ++u) acc[h] |= v[h][u];
  }
#pragma unroll
  for (int h = 0; h < kHeads; ++h)
    for (int s = width; s < 32; s <<= 1) acc[h] |= __shfl_xor_sync(0xffffffffu, acc[h], s);
}

template <bool kLong>
__global__ void __launch_bounds__(kUnionThreads) union_count_kernel(const uint32_t* __restrict__ mask,
                                                                    const int32_t* __restrict__ rank, int H, int NB,
                                                                    int Wd, int P, uint32_t* __restrict__ U,
                                                                    int include_local, int32_t* __restrict__ cnt,
                                                                    int32_t* __restrict__ received,
                                                                    int32_t* __restrict__ n_src) {
  enter_grid(mask, rank);
  __shared__ uint32_t own_s[kMaxRanks * kMaxWords];
  __shared__ uint32_t u_s[kMaxWords];
  __shared__ uint16_t rows_s[kMaxBlocks];
  __shared__ int n_rows_s;
  const int r = blockIdx.x % P, bh = blockIdx.x / P, bb = bh / H, h = bh % H;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = kUnionThreads / 32;
  if (threadIdx.x == 0) n_rows_s = 0;
  if (threadIdx.x < kMaxWords) u_s[threadIdx.x] = 0u;
  if (blockIdx.x == 0 && threadIdx.x == 0 && n_src) *n_src = 0;
  const uint32_t* m = mask + (int64_t)bh * NB * Wd;
  const int width = lanes_per_row(Wd);
  uint32_t acc = 0;
  if constexpr (kLong) {
    for (int i = threadIdx.x; i < P * Wd; i += kUnionThreads) own_s[i] = 0u;
    const int n_rows = list_rows(rank, NB, Wd, P, r, own_s, rows_s);
    uint32_t all[1];
    or_rows<1, 8>(m, 0, 1, rows_s, n_rows, Wd, width, all);
    acc = all[0];
  } else {
    own_words(rank, NB, Wd, P, own_s);
    for (int i = threadIdx.x; i < NB; i += kUnionThreads)
      if (rank[i] == r) rows_s[atomicAdd(&n_rows_s, 1)] = (uint16_t)i;
    __syncthreads();
    const int n_rows = n_rows_s, per_warp = 32 / width, w = lane & (width - 1);
#pragma unroll 4
    for (int k = warp * per_warp + lane / width; k < n_rows; k += n_warps * per_warp)
      if (w < Wd) acc |= m[(int64_t)rows_s[k] * Wd + w];
    for (int s = width; s < 32; s <<= 1) acc |= __shfl_xor_sync(0xffffffffu, acc, s);
  }
  if (lane < Wd && acc) atomicOr(&u_s[lane], acc);
  __syncthreads();
  const uint32_t u = lane < Wd ? u_s[lane] : 0u;
  if (warp == 0 && lane < Wd) U[((int64_t)(bb * P + r) * H + h) * Wd + lane] = u;
  for (int p = warp; p < P; p += n_warps) {
    const int c = __reduce_add_sync(0xffffffffu, lane < Wd ? __popc(u & own_s[p * Wd + lane]) : 0);
    if (lane == 0) cnt[((int64_t)(bb * P + r) * P + p) * H + h] = c;
  }
  if (received && warp == n_warps - 1) {  // (up to 15 ranks this warp has no counts to take)
    uint32_t packed = 0;
    if (lane < Wd)
      for (int p = 0; p < P; ++p) packed |= p != r || include_local ? own_s[p * Wd + lane] : 0u;
    const int c = __reduce_add_sync(0xffffffffu, __popc(u & packed));
    if (lane == 0) received[(int64_t)(bb * P + r) * H + h] = c;
  }
}

// Unions, counts and offsets of a plan without destinations, in one launch: a cluster of CTAs per consumer takes the
// consumer's heads in turn, meets when all counts are there, and its first CTA scans them.  Nothing is kept between
// launches.  Latency-bound, and what is saved is the host's time for a launch.  us a plan with two launches / this way,
// one call behind the other and in a graph, where the host is out of it: 2 heads x 64 blocks, 4 ranks 7.4 / 5.1 and 4.0
// / 3.8; 4 x 1000, 8 ranks 7.6 / 5.1 and 5.6 / 4.4; 13 x 77, 5 ranks 7.6 / 5.4 and 4.3 / 4.3; 24 x 384, 4 ranks 8.2 /
// 5.3 and 4.9 / 4.4; 24 x 300, 11 ranks 7.9 / 5.4 and 6.1 / 6.0; 16 x 500, 2 ranks 7.7 / 5.2 and 4.4 / 5.2.  Beyond the
// line 24 x 929, 8 ranks (10530 words a CTA) 7.6 / 6.8 and 5.8 / 6.5, 12 x 600, 2 ranks (11400) 7.5 / 7.3 and 5.3 /
// 7.1, 9 x 1000, 3 ranks (21376) 7.5 / 8.0 and 5.5 / 7.8.  (The heads of a CTA one after the other: 24 x 384 5.8 and
// 5.5, 21 x 22, 7 ranks 6.1 and 5.4, now 5.3 and 4.9.)
constexpr int kPlanCtas = 8, kPlanHeads = 3;  // CTAs of a cluster, heads that one takes
constexpr int kPlanWords = 10240;             // mask words of two or three heads
static bool plan_fits_clusters(const Geometry& g, int P, int sms) {
  const int ctas = std::min(g.H, kPlanCtas), heads = (g.H + ctas - 1) / ctas, rows = (g.NB + P - 1) / P;
  return heads <= kPlanHeads && (heads == 1 || heads * rows * g.Wd <= kPlanWords) && g.H * P <= kUnionThreads &&
         g.B * P * ctas <= sms;
}

__global__ void __launch_bounds__(kUnionThreads)
    cluster_plan_kernel(const uint32_t* __restrict__ mask, const int32_t* __restrict__ rank, int H, int NB, int Wd,
                        int P, uint32_t* __restrict__ U, int include_local, int32_t* __restrict__ cnt,
                        int64_t* __restrict__ seg_off, int64_t* __restrict__ seg_total, int64_t* __restrict__ volume,
                        int64_t entry_bytes) {
  enter_grid(mask, rank);
  __shared__ uint32_t own_s[kMaxRanks * kMaxWords];
  __shared__ uint32_t u_s[kPlanHeads][kMaxWords];
  __shared__ uint16_t rows_s[kMaxBlocks];
  const int ctas = min(H, kPlanCtas), br = blockIdx.x / ctas, bb = br / P, r = br - bb * P;
  const int h0 = blockIdx.x - br * ctas, n_heads = (H - h0 + ctas - 1) / ctas;  // heads h0, h0 + ctas, ...
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int n_warps = kUnionWarps;
  for (int i = threadIdx.x; i < kPlanHeads * kMaxWords; i += kUnionThreads) (&u_s[0][0])[i] = 0u;
  for (int i = threadIdx.x; i < P * Wd; i += kUnionThreads) own_s[i] = 0u;
  const int n_rows = list_rows(rank, NB, Wd, P, r, own_s, rows_s);
  const int width = lanes_per_row(Wd);
  const uint32_t* m = mask + (int64_t)(bb * H + h0) * NB * Wd;
  const int64_t pitch = (int64_t)ctas * NB * Wd;
  if (n_heads == 1) {
    uint32_t acc[1];
    or_rows<1, 8>(m, pitch, 1, rows_s, n_rows, Wd, width, acc);
    if (lane < Wd && acc[0]) atomicOr(&u_s[0][lane], acc[0]);
  } else {
    uint32_t acc[kPlanHeads];
    or_rows<kPlanHeads, 4>(m, pitch, n_heads, rows_s, n_rows, Wd, width, acc);
#pragma unroll
    for (int k = 0; k < kPlanHeads; ++k)
      if (lane < Wd && acc[k]) atomicOr(&u_s[k][lane], acc[k]);
  }
  __syncthreads();
  for (int i = warp; i < n_heads * P; i += n_warps) {
    const int k = i / P, p = i - k * P, h = h0 + k * ctas;
    const uint32_t u = lane < Wd ? u_s[k][lane] : 0u;
    if (p == 0 && lane < Wd) U[((int64_t)br * H + h) * Wd + lane] = u;
    const int c = __reduce_add_sync(0xffffffffu, lane < Wd ? __popc(u & own_s[p * Wd + lane]) : 0);
    if (lane == 0) cnt[((int64_t)br * P + p) * H + h] = c;
  }
  asm volatile("barrier.cluster.arrive.aligned;\n\tbarrier.cluster.wait.aligned;" ::: "memory");
  if (h0 != 0) return;
  // the consumer's counts in pack order, one per thread
  __shared__ int sum_s[n_warps], remote_s[n_warps];
  const int i = (int)threadIdx.x, n = P * H;
  const int c = i < n ? __ldcg(cnt + (int64_t)br * n + i) : 0;
  const bool local = i / H == r;
  const int counted = local && !include_local ? 0 : c, remote = __reduce_add_sync(0xffffffffu, local ? 0 : c);
  int incl = counted;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, s);
    if (lane >= s) incl += v;
  }
  if (lane == 31) {
    sum_s[warp] = incl;
    remote_s[warp] = remote;
  }
  __syncthreads();
  int first = 0, all = 0, all_remote = 0;
#pragma unroll
  for (int k = 0; k < n_warps; ++k) {
    first += k < warp ? sum_s[k] : 0;
    all += sum_s[k];
    all_remote += remote_s[k];
  }
  if (i < n) seg_off[(int64_t)br * n + i] = first + incl - counted;
  if (i == 0) {
    seg_total[br] = all;
    volume[br] = entry_bytes * all_remote;
  }
}

// Pack-order offsets, and where every packed tile goes.  A CTA per consumer scans its consumer's counts in pack
// order (producer, then head) and writes offsets, total and volume.  With `dst` given there are consumers + batch items
// CTAs per `heads` heads: CTA (consumer, h) also fills its column of the destination table
//   dst[(b*H + h)*NB + j][r] = byte offset in `packed` of consumer r's copy of block j, or -1
// one warp per producer (the consumer's base is its caller-given dst_base or the sum of `received` over all earlier
// consumers), and CTA (B*P + b, h) appends the blocks that any consumer of batch item b receives to the list of
// sources, a head's blocks together.  The order of the heads in that list is the order in which they arrive; it decides
// nothing but the order of the copies.
// Latency-bound integer work on a few MB, so every CTA repeats the scan (P*H counts) and the sum (at most B*P*H values)
// rather than wait for another launch.  (A serial scan per consumer in one CTA and a launch for the entries: 13 + 7 us
// on 24 heads, 8 ranks, 18 + 4 us on 48 heads; offsets alone 2 us now, with destinations 9 us on 48 and 15 us on 24
// heads; eight heads to a CTA, one warp each: 16-19 us.  Union, plan and an empty gather at the limit, 16 batch items x
// 64 ranks x 24 heads: 0.55 ms; 72 ms with the sum over the counts of every producer, 2.9 ms with the serial scan.)
// A CTA takes one head up to 64 heads, and so many beyond that there are about 64 CTAs per consumer: the scans repeated
// per head would grow with the square of the heads (plan and gather of 2000 heads x 4 blocks, 8 ranks: 184 us, 1447
// with a head per CTA, 731 with the serial scan; 300 heads x 20 blocks 34, 63 and 122).
constexpr int kPlanThreads = 256;
constexpr int kPlanMaxHeads = 32;

static int plan_heads(int H) { return H <= 64 ? 1 : std::min(kPlanMaxHeads, (H + 63) / 64); }

__device__ __forceinline__ int64_t block_sum(int64_t v, int64_t* warp_s) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) v += __shfl_xor_sync(0xffffffffu, v, s);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) warp_s[threadIdx.x >> 5] = v;
  __syncthreads();
  int64_t t = 0;
#pragma unroll
  for (int k = 0; k < kPlanThreads / 32; ++k) t += warp_s[k];
  return t;
}

__global__ void __launch_bounds__(kPlanThreads) plan_kernel(
    const int32_t* __restrict__ cnt, const int32_t* __restrict__ received, const uint32_t* __restrict__ U,
    const int32_t* __restrict__ rank, int BP, int H, int heads, int NB, int Wd, int P, int include_local,
    int64_t entry_bytes, int64_t* __restrict__ seg_off, int64_t* __restrict__ seg_total,
    int64_t* __restrict__ volume, const int64_t* __restrict__ dst_base, int64_t capacity, int64_t* __restrict__ dst,
    int32_t* __restrict__ src, int32_t* __restrict__ n_src, int32_t* __restrict__ status) {
  enter_grid(cnt, received, U, rank, dst_base);
  __shared__ uint32_t own_s[kMaxRanks * kMaxWords];
  extern __shared__ int64_t seg_s[];  // [heads][P] first entry of (my head, producer)
  __shared__ int64_t warp_s[kPlanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_x = BP + (dst ? BP / P : 0), x = blockIdx.x % n_x;
  const int h0 = blockIdx.x / n_x * heads, h1 = min(h0 + heads, H);  // my heads
  if (dst) own_words(rank, NB, Wd, P, own_s);
  if (x >= BP) {  // the blocks of my heads that any consumer receives, a warp per head
    __syncthreads();
    const int bb = x - BP;
    for (int h = h0 + warp; h < h1; h += kPlanThreads / 32) {
      uint32_t live = 0, owned = 0;
      if (lane < Wd) {
        for (int p = 0; p < P; ++p) owned |= own_s[p * Wd + lane];
#pragma unroll 8
        for (int r = 0; r < P; ++r)
          live |= U[((int64_t)(bb * P + r) * H + h) * Wd + lane] &
                  (include_local ? owned : owned & ~own_s[r * Wd + lane]);
      }
      int total, first = 0;
      int at = bits_below(live, lane, &total);
      if (lane == 0) first = atomicAdd(n_src, total);
      at += __shfl_sync(0xffffffffu, first, 0);
      for (; live; live &= live - 1) src[at++] = (bb * H + h) * NB + lane * 32 + __ffs(live) - 1;
    }
    return;
  }

  const int br = x, bb = br / P, r = br % P;
  const int PH = P * H;
  const bool writer = h0 == 0;
  const int32_t* mine = cnt + (int64_t)br * PH;
  int64_t cursor = 0, remote = 0;  // entries of earlier chunks of this consumer
  for (int i0 = 0; i0 < PH; i0 += kPlanThreads) {
    const int i = i0 + (int)threadIdx.x;
    const int c = i < PH ? mine[i] : 0;
    const int p = i / H;
    const int counted = p != r || include_local ? c : 0;
    if (p != r) remote += c;
    int incl = counted;  // a chunk holds at most kPlanThreads * kMaxBlocks entries
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, s);
      if (lane >= s) incl += v;
    }
    __syncthreads();  // (the previous chunk's sums have been read)
    if (lane == 31) warp_s[warp] = incl;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int k = 0; k < kPlanThreads / 32; ++k) {
      const int v = (int)warp_s[k];
      if (k < warp) before += v;
      all += v;
    }
    if (i < PH) {
      const int64_t at = cursor + before + incl - counted;
      if (writer) seg_off[(int64_t)br * PH + i] = at;
      const int h = i - p * H;
      if (h >= h0 && h < h1) seg_s[(h - h0) * P + p] = at;
    }
    cursor += all;
  }
  if (writer) {
    remote = block_sum(remote, warp_s);
    if (threadIdx.x == 0) {
      seg_total[br] = cursor;
      volume[br] = entry_bytes * remote;
    }
  }
  if (!dst) return;

  int64_t base = 0;
  if (dst_base) {
    base = dst_base[br];
  } else if (br > 0) {
    int64_t n = 0;
    for (int k = threadIdx.x; k < br * H; k += kPlanThreads) n += received[k];
    base = entry_bytes * block_sum(n, warp_s);
  }
  for (int h = h0; h < h1; ++h) {
    int64_t* out = dst + (int64_t)(bb * H + h) * NB * P + r;
    const uint32_t u = lane < Wd ? U[((int64_t)br * H + h) * Wd + lane] : 0u;
    for (int j = threadIdx.x; j < NB; j += kPlanThreads) out[(int64_t)j * P] = -1;
    __syncthreads();
    for (int p = warp; p < P; p += kPlanThreads / 32) {
      if (p == r && !include_local) continue;
      uint32_t bits = lane < Wd ? u & own_s[p * Wd + lane] : 0u;
      int total;
      int64_t byte = base + (seg_s[(h - h0) * P + p] + bits_below(bits, lane, &total)) * entry_bytes;
      for (; bits; bits &= bits - 1, byte += entry_bytes) {
        if (capacity >= 0 && byte + entry_bytes > capacity) {
          atomicExch(status, SPARSP_ERR_CAPACITY);  // would overflow: stays -1, the gather leaves it out
        } else {
          out[(int64_t)(lane * 32 + __ffs(bits) - 1) * P] = byte;
        }
      }
    }
  }
}

// Table of destinations [B*H*NB][n_dst] and list of sources [<= B*H*NB] inside the workspace's entry area, which holds
// 16 bytes for every (source, rank).
static int64_t* dst_table(char* ws, const WsLayout& L) { return (int64_t*)(ws + L.entries); }
static int32_t* src_list(char* ws, const WsLayout& L, const Geometry& g, int n_dst) {
  return (int32_t*)(ws + L.entries + (int64_t)g.B * g.H * g.NB * n_dst * 8);
}
// Entries per (consumer, head) [B*P*H] behind them: tables and list take 8 P + 4 of the 16 P bytes for a block, these 4
// P for a head.
static int32_t* received_table(char* ws, const WsLayout& L, const Geometry& g, int P) {
  return src_list(ws, L, g, P) + (int64_t)g.B * g.H * g.NB;
}

static cudaError_t launch_union(const Geometry& g, const uint32_t* mask, const int32_t* rank, int P, int include_local,
                                uint32_t* U, int32_t* cnt, int32_t* received, int32_t* n_src, cudaStream_t st) {
  auto kern = rows_are_long(g, P) ? union_count_kernel<true> : union_count_kernel<false>;
  return launch_kernel(kern, g.B * g.H * P, kUnionThreads, 0, st, mask, rank, g.H, g.NB, g.Wd, P, U,
                       include_local, cnt, received, n_src);
}

// dst, src, n_src, received: NULL for a plan without destinations.
static cudaError_t launch_plan(const Geometry& g, const uint32_t* mask, const int32_t* rank, int P, int include_local,
                               uint32_t* U, int32_t* cnt, int64_t* seg_off, int64_t* seg_total, int64_t* volume,
                               const int64_t* dst_base, int64_t capacity, int64_t* dst, int32_t* src, int32_t* n_src,
                               int32_t* received, int32_t* status, cudaStream_t st) {
  const cudaError_t e = launch_union(g, mask, rank, P, include_local, U, cnt, received, n_src, st);
  if (e != cudaSuccess) return e;
  const int heads = dst ? plan_heads(g.H) : 1;
  const unsigned grid = dst ? (unsigned)((g.B * P + g.B) * ((g.H + heads - 1) / heads)) : (unsigned)(g.B * P);
  return launch_kernel(plan_kernel, grid, kPlanThreads, (size_t)heads * P * 8, st, cnt, received, U, rank, g.B * P, g.H,
                       heads, g.NB, g.Wd, P, include_local, 2LL * g.b * g.d * 2, seg_off, seg_total, volume, dst_base,
                       capacity, dst, src, n_src, status);
}

static int check_consumers(const Geometry& g, int P) {
  if (g.B * P <= 1024) return SPARSP_OK;
  set_error("batch * n_ranks = %d exceeds 1024", g.B * P);
  return SPARSP_ERR_UNSUPPORTED;
}

int launch_demand(const Geometry& g, const uint32_t* mask, const int32_t* rank_of_block, int P, int flags, uint32_t* U,
                  int32_t* cnt, int64_t* seg_off, int64_t* seg_total, int64_t* volume, char* ws, const WsLayout& L,
                  cudaStream_t st) {
  const int rc = check_consumers(g, P);
  if (rc != SPARSP_OK) return rc;
  const int local = (flags & SPARSP_INCLUDE_LOCAL) ? 1 : 0, ctas = std::min(g.H, kPlanCtas);
  int sms = 0;
  SPARSP_CUDA_OK(sm_count(&sms));
  if (plan_fits_clusters(g, P, sms)) {
    SPARSP_CUDA_OK(launch_clusters(cluster_plan_kernel, g.B * P * ctas, ctas, kUnionThreads, 0, st, mask, rank_of_block,
                                   g.H, g.NB, g.Wd, P, U, local, cnt, seg_off, seg_total, volume, 2LL * g.b * g.d * 2));
    return SPARSP_OK;
  }
  SPARSP_CUDA_OK(launch_plan(g, mask, rank_of_block, P, local, U, cnt, seg_off, seg_total, volume, nullptr, -1, nullptr,
                             nullptr, nullptr, nullptr, (int32_t*)(ws + L.status), st));
  return SPARSP_OK;
}

// ------------------------------------------------------------------------------------------------
// Gather, source by source: a K or V tile is loaded into shared memory once and stored from there to every consumer
// that selected it, so HBM carries one read per distinct tile and one write per packed tile -- its floor.  (Tile by
// tile in the order of the packed buffer every copy was read again: 3.45 ms for the 10.8 GB that 8 ranks of 40 heads x
// 591 blocks of 32 KiB receive, at 6.3 TB/s of reads and writes; this order 2.23 ms, 5.5 TB/s of which seven eighths
// are writes.  Four to six stages and one to three stores left in flight are within 1 %: memory sets the pace.)
// One warp streams whole tiles: TMA tile load (any token stride; rows behind the last token arrive as zeros), then one
// bulk store per consumer, issued by the lane that holds its destination.  A ring of kPackStages tile buffers per warp
// (1, 2 or 4 warps per CTA for 32, 16, 8 KiB tiles: 160 KiB per CTA whatever the tile size), loads running
// kPackStages - 1 tiles ahead of the stores.  The warp's next 32 sources sit in its lanes' registers and the next
// tile's destinations are fetched before the wait for the current stores, so that no table lookup is exposed.
// ------------------------------------------------------------------------------------------------
constexpr int kPackStages = 5;
constexpr int kPackMaxWarps = 4;

// Nobody reads the copies before a consumer fetches them, so the L2 cache need not keep them: the sources, which are
// read again for other consumers, and K and V stay there longer (demand and gather of 24 heads x 24576 226.5 -> 224 us,
// of 48 x 17776 328.5 -> 325.5, of 40 x 75600 2221 -> 2207; seven segments 394.7 -> 392).
__device__ __forceinline__ void bulk_store(void* gdst, const void* smem_src, uint32_t bytes) {
  uint64_t policy;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(policy));
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group.L2::cache_hint [%0], [%1], %2, %3;" ::"l"(gdst),
               "r"(ptx::smem_u32(smem_src)), "r"(bytes), "l"(policy)
               : "memory");
}

__global__ void __launch_bounds__(32 * kPackMaxWarps) pack_kernel(const __grid_constant__ CUtensorMap tmK,
                                                                  const __grid_constant__ CUtensorMap tmV,
                                                                  const int64_t* __restrict__ dst, int n_dst,
                                                                  const int32_t* __restrict__ src,
                                                                  const int32_t* __restrict__ n_src, int H, int NB,
                                                                  int b, uint32_t tile_bytes,
                                                                  unsigned char* __restrict__ packed,
                                                                  int32_t* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ uint64_t full_all[kPackMaxWarps * kPackStages];
  __shared__ int s_abort;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n_warps = blockDim.x >> 5;
  uint64_t* full = full_all + warp * kPackStages;
  unsigned char* ring = smem_raw + (size_t)warp * kPackStages * tile_bytes;  // this warp's buffers
  const int unit = blockIdx.x * n_warps + warp, n_units = gridDim.x * n_warps;
  if (threadIdx.x == 0) s_abort = 0;
  if (lane == 0) {
    for (int st = 0; st < kPackStages; ++st) ptx::mbar_init(full + st, 1);
    ptx::mbar_init_fence();
  }
  enter_grid(dst, src, n_src);
  __syncthreads();
  const int64_t n_items = 2 * (int64_t)*n_src;  // item: K (even) or V (odd) tile of source item / 2
  const int n_local = (int)(n_items > unit ? (n_items - unit + n_units - 1) / n_units : 0);

  // lane l: the source of local item q + l
  auto sources = [&](int q) -> int {
    const int64_t item = unit + (int64_t)(q + lane) * n_units;
    return item < n_items ? __ldg(src + (item >> 1)) : 0;
  };
  auto which = [&](int q) { return (int)((unit + (int64_t)q * n_units) & 1); };
  auto destination = [&](int s, int first) -> int64_t {
    return first + lane < n_dst ? __ldg(dst + (int64_t)s * n_dst + first + lane) : -1;
  };
  auto issue_load = [&](int q, int s) {
    uint64_t* bar = full + q % kPackStages;
    const int bh = s / NB;
    ptx::mbar_expect_tx(bar, tile_bytes);
    ptx::tma_load_4d(ring + (size_t)(q % kPackStages) * tile_bytes, which(q) ? &tmV : &tmK, bar, 0, (s - bh * NB) * b,
                     bh % H, bh / H);
  };
  int cur = sources(0), ahead = cur;  // sources of the 32 items around the store / around the load
  for (int q = 0; q < kPackStages - 1 && q < n_local; ++q) {
    const int s = __shfl_sync(0xffffffffu, ahead, q);
    if (lane == 0) issue_load(q, s);
  }
  int64_t d0 = -1, d1 = -1;  // this lane's destinations of the current item (ranks lane and lane + 32)
  if (n_local > 0) {
    const int s = __shfl_sync(0xffffffffu, cur, 0);
    d0 = destination(s, 0);
    if (n_dst > 32) d1 = destination(s, 32);
  }
  for (int q = 0; q < n_local; ++q) {
    const int64_t half = which(q) ? tile_bytes : 0;
    const unsigned char* buf = ring + (size_t)(q % kPackStages) * tile_bytes;
    ptx::mbar_wait_bounded(full + q % kPackStages, (uint32_t)((q / kPackStages) & 1), &s_abort, status, 50,
                           200000000LL);
    if (d0 >= 0) bulk_store(packed + d0 + half, buf, tile_bytes);
    if (d1 >= 0) bulk_store(packed + d1 + half, buf, tile_bytes);
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    if (q + 1 < n_local) {
      if (((q + 1) & 31) == 0) cur = sources(q + 1);
      const int s = __shfl_sync(0xffffffffu, cur, (q + 1) & 31);
      d0 = destination(s, 0);
      if (n_dst > 32) d1 = destination(s, 32);
    }
    const int ql = q + kPackStages - 1;
    if (ql < n_local) {
      if ((ql & 31) == 0) ahead = sources(ql);
      const int s = __shfl_sync(0xffffffffu, ahead, ql & 31);
      // the buffer of item q - 1 may be refilled once every lane's stores have read it
      asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
      __syncwarp();
      if (lane == 0) issue_load(ql, s);
    }
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Tensor maps and grid of a kernel that moves tiles as pack_kernel does, and its shared memory.
struct PackLaunch {
  CUtensorMap tk, tv;
  unsigned grid;
  uint32_t tile_bytes;
};
static int pack_warps(int tile_bytes) { return std::max(1, std::min(kPackMaxWarps, (32 * 1024) / tile_bytes)); }
static int prepare_pack(const sparsp_shape& s, const Geometry& g, const void* K, const void* V, const void* kernel,
                        int smem, PackLaunch* c) {
  int sms = 0;
  SPARSP_CUDA_OK(sm_count(&sms));
  int rc;
  if ((rc = make_tile_tmap(&c->tk, K, s, g, g.b, false)) != SPARSP_OK) return rc;
  if ((rc = make_tile_tmap(&c->tv, V, s, g, g.b, false)) != SPARSP_OK) return rc;
  c->tile_bytes = (uint32_t)(g.b * g.d * 2);
  c->grid = (unsigned)sms;
  SPARSP_CUDA_OK(ensure_dynamic_smem(kernel, smem));
  return SPARSP_OK;
}

// ------------------------------------------------------------------------------------------------
// Offsets and gather in one launch, for plans of up to kScanMax counts: every CTA scans the counts of all consumers
// into shared memory (their flat order is the order of the packed buffers), and a copy's place is its segment's first
// entry plus the blocks of the segment below it, counted in the union words by the lane of its consumer.  The other
// half of its warps meanwhile numbers the blocks that anybody receives, of all heads, so that only those are handed
// out.  No tables, no list of sources in memory and no launch that makes them.  The first CTAs also write the offsets,
// totals and volumes.  Tiles move as in pack_kernel, a block's K and V together (an entry is one store), kGatherStages
// - 1 blocks of loads in flight.  us of the whole call with tables and the n-th source of the list for the n-th warp /
// this way: 40 heads x 75600, 8 ranks 2176 / 1931 (6.4 TB/s), 24 x 118800 1714 / 1522, 48 x 17776 322 / 287, 24 x
// 24576, 4 ranks 223 / 200, 2 x 13 x 6034, 3 ranks 18.0 / 13.9, 2 x 4096 18.3 / 10.3.  What held it back was not memory
// but warps whose blocks happened to have many consumers.  Where little is wanted, with tables / this way / with every
// block handed out and looked up, wanted or not: 40 heads x 591 blocks of 128 x 128, a band of two blocks either side,
// 8 ranks 38 / 38 / 158, one rank 12.6 / 11 / 96, two heads of all 129 / 115 / 231.
// The counts, the words of live blocks and a table of owners have to fit beside the rings, and every CTA scans all of
// them: a few us at 6144 counts (24 heads, 16 ranks 1712 / 1483; one more head, by tables, 1784 / 1770).
// ------------------------------------------------------------------------------------------------
constexpr int kScanMax = 6144;
// Masks of up to kMaskMax words are read by every CTA, which makes the unions and counts for itself (kFromMask): no
// launch of the union before it.  A warp then gets every n-th block, of which there are few enough for that.  us of the
// whole call with the union's launch / without: 2 heads x 64 blocks, 4 ranks 10.2 / 8.1; 7 x 21 of d = 128, 7 ranks
// 11.5 / 8.5; 48 x 13 of 128 x 128, 7 ranks 27.0 / 23.0; 2 x 13 x 48, 3 ranks 13.3 / 11.6; 40 x 40, 8 ranks 29.9 / 28.4
// (3200 words); beyond the line 24 x 80 (5760 words) 20.2 / 22.7, 9 x 166 (8964) 27.9 / 31.2; 16 x 64 of 128 x 128 in 7
// blocks a warp 43.8 / 44.3.  Between four and six blocks a warp only with 2560 words at most: 13 x 60 of 128 x 128, 4
// ranks (1560 words) 38.2 / 36.3, 9 x 80, 5 ranks (2160) 41.0 / 40.6, 2 x 13 x 48 of 64 x 128 (2496), but 5 x 144, 14
// ranks (3600) 78.3 / 81.1, 7 x 120, 8 ranks (3360) 69.0 / 72.5, 22 x 64 of 64 x 128 (2816) 47.5 / 50.0.
constexpr int kMaskMax = 4096, kMaskMaxMany = 2560, kFromMaskBlocks = 6, kFromMaskFew = 4;
constexpr int kGatherStages = 3, kGatherThreads = 512;
constexpr int kGatherSmem = 232448 - 7 * 1024;  // dynamic shared memory, next to less than 7 KB of its own

// out[i] = sum of value(0 .. i - 1) for i <= n, in two steps with a barrier between them and one behind: n_warps warps,
// of which this one is `warp`, scan a part each, then add what lies before it.
template <int kUnroll, typename F>
__device__ __forceinline__ void scan_part(int n, int warp, int n_warps, int32_t* out, int* warp_s, F value) {
  const int lane = threadIdx.x & 31;
  const int chunk = (n + 32 * n_warps - 1) / (32 * n_warps) * 32;
  const int i1 = min(n, (warp + 1) * chunk);
  int running = 0;
#pragma unroll kUnroll
  for (int i0 = warp * chunk; i0 < i1; i0 += 32) {
    const int i = i0 + lane;
    const int c = i < i1 ? value(i) : 0;
    int incl = c;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, s);
      if (lane >= s) incl += v;
    }
    if (i < i1) out[i] = running + incl - c;
    running += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) warp_s[warp] = running;
}
__device__ __forceinline__ void scan_rest(int n, int warp, int n_warps, int32_t* out, const int* warp_s) {
  const int lane = threadIdx.x & 31;
  const int chunk = (n + 32 * n_warps - 1) / (32 * n_warps) * 32;
  const int i1 = min(n, (warp + 1) * chunk);
  int before = 0, all = 0;
  for (int k = 0; k < n_warps; ++k) {
    before += k < warp ? warp_s[k] : 0;
    all += warp_s[k];
  }
  for (int i = warp * chunk + lane; i < i1; i += 32) out[i] += before;
  if (warp == 0 && lane == 0) out[n] = all;
}

template <bool kFromMask>
__global__ void __launch_bounds__(kGatherThreads)
    gather_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                  const uint32_t* __restrict__ mask, uint32_t* __restrict__ U_out, const int32_t* __restrict__ rank,
                  int32_t* __restrict__ cnt_out, int B,
                  int H, int NB, int Wd, int P, int include_local, int b, uint32_t tile_bytes, int n_copy,
                  int64_t* __restrict__ seg_off, int64_t* __restrict__ seg_total, int64_t* __restrict__ volume,
                  const int64_t* __restrict__ dst_base, int64_t capacity, unsigned char* __restrict__ packed,
                  int32_t* __restrict__ n_taken, int32_t* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ uint64_t full_all[kPackMaxWarps * kGatherStages];
  __shared__ int64_t dst_all[kPackMaxWarps][kGatherStages][kMaxRanks];
  __shared__ int warp_s[kGatherThreads / 32];
  __shared__ int s_abort;
  static_assert(sizeof(full_all) + sizeof(dst_all) + sizeof(warp_s) + sizeof(s_abort) + 128 <= 232448 - kGatherSmem,
                "shared memory budget");
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int PH = P * H, T = B * P * PH, n_words = B * H * Wd;
  const int64_t entry_bytes = 2LL * tile_bytes;
  int32_t* off_s = reinterpret_cast<int32_t*>(smem_raw + (size_t)n_copy * kGatherStages * entry_bytes);  // [T + 1]
  int32_t* pos_s = off_s + T + 1;                                        // [n_words + 1] live blocks before each word's
  uint32_t* live_s = reinterpret_cast<uint32_t*>(pos_s + n_words + 1);   // [B*H][Wd] blocks that any consumer receives
  uint32_t* own_s = live_s + n_words;                                    // [P][Wd]
  uint32_t* union_s = own_s + P * Wd;                                    // kFromMask: [B*P][H][Wd]
  if (threadIdx.x == 0) s_abort = 0;
  if (threadIdx.x < kPackMaxWarps * kGatherStages) {
    ptx::mbar_init(full_all + threadIdx.x, 1);
    ptx::mbar_init_fence();
  }
  // The launches behind this one begin when its CTAs end: an attention that takes its places while CTAs are still
  // copying makes the step longer (mask, demand and gather, attention of 2 x 13 x 6034 tokens 138 us, 131 this way, 141
  // with the gather by tables; of 2 x 4096 39.2, 38.8 and 41).
  const uint32_t* U = U_out;
  const int32_t* cnt = cnt_out;
  wait_previous_grids(mask, U, rank, cnt, dst_base);
  if (kFromMask)
    for (int i = threadIdx.x; i < n_words * P; i += kGatherThreads) union_s[i] = 0u;
  own_words(rank, NB, Wd, P, own_s);
  if (kFromMask) {
    const int n_mask = B * H * NB * Wd;
    constexpr int kFlight = 8;
    for (int i0 = threadIdx.x; i0 < n_mask; i0 += kFlight * kGatherThreads) {
      uint32_t v[kFlight];
#pragma unroll
      for (int u = 0; u < kFlight; ++u) v[u] = i0 + u * kGatherThreads < n_mask ? mask[i0 + u * kGatherThreads] : 0u;
#pragma unroll
      for (int u = 0; u < kFlight; ++u) {
        if (v[u] == 0u) continue;
        const int i = i0 + u * kGatherThreads, row = i / Wd, w = i - row * Wd, bh = row / NB, bb = bh / H;
        const int r = rank[row - bh * NB];
        if ((unsigned)r < (unsigned)P) atomicOr(&union_s[((bb * P + r) * H + bh - bb * H) * Wd + w], v[u]);
      }
    }
    U = union_s;
  }
  __syncthreads();
  if (kFromMask)
    for (int i = blockIdx.x * kGatherThreads + threadIdx.x; i < n_words * P; i += gridDim.x * kGatherThreads)
      U_out[i] = union_s[i];
  // One half of the warps scans the counts, the other the words of live blocks.
  constexpr int kHalf = kGatherThreads / 64;
  if (warp < kHalf) {
    scan_part<4>(T, warp, kHalf, off_s, warp_s, [&](int i) {
      const int br = i / PH, q = (i - br * PH) / H;
      int c;
      if (kFromMask) {
        const uint32_t* u = U + ((int64_t)br * H + i % H) * Wd;
        c = 0;
        for (int w = 0; w < Wd; ++w) c += __popc(u[w] & own_s[q * Wd + w]);
        if (blockIdx.x == 0) cnt_out[i] = c;
      } else {
        c = cnt[i];
      }
      return q != br % P || include_local ? c : 0;
    });
  } else {
    scan_part<1>(n_words, warp - kHalf, kHalf, pos_s, warp_s + kHalf, [&](int i) {
      const int bh = i / Wd, w = i - bh * Wd, bb = bh / H;
      const uint32_t* u = U + ((int64_t)bb * P * H + bh - bb * H) * Wd + w;
      uint32_t live = 0, owned = 0;
#pragma unroll 8
      for (int r = 0; r < P; ++r) {
        const uint32_t own = own_s[r * Wd + w];
        live |= u[(int64_t)r * H * Wd] & (include_local ? ~0u : ~own);
        owned |= own;
      }
      live_s[i] = live & owned;
      return __popc(live & owned);
    });
  }
  __syncthreads();
  if (warp < kHalf) scan_rest(T, warp, kHalf, off_s, warp_s);
  else scan_rest(n_words, warp - kHalf, kHalf, pos_s, warp_s + kHalf);
  __syncthreads();
  for (int br = blockIdx.x; br < B * P; br += gridDim.x) {
    const int first = off_s[br * PH], total = off_s[(br + 1) * PH] - first, own = (br % P) * H;
    for (int i = threadIdx.x; i < PH; i += kGatherThreads) seg_off[(int64_t)br * PH + i] = off_s[br * PH + i] - first;
    if (threadIdx.x == 0) {
      seg_total[br] = total;
      volume[br] = entry_bytes * (total - (off_s[br * PH + own + H] - off_s[br * PH + own]));
    }
  }
  if (warp >= n_copy) return;

  uint64_t* full = full_all + warp * kGatherStages;
  unsigned char* ring = smem_raw + (size_t)warp * kGatherStages * entry_bytes;
  int64_t(*dst_s)[kMaxRanks] = dst_all[warp];
  const int n_units = gridDim.x * n_copy;
  // Blocks are copied to between one and all consumers, so a warp takes its next one, a number among those that anybody
  // receives, from a counter, and the number after that while it looks the block up.
  int next = blockIdx.x * n_copy + warp;
  const int n_blocks = pos_s[n_words];
  int word = 0;  // the one that holds the last block taken (numbers only grow)
  // where consumer r's copy of block j goes, -1 if it gets none
  auto destination = [&](int bb, int h, int j, int p, int r) -> int64_t {
    if (r == p && !include_local) return -1;
    const int br = bb * P + r;
    const uint32_t* u = U + ((int64_t)br * H + h) * Wd;
    const uint32_t* own = own_s + p * Wd;
    const int w = j >> 5;
    const uint32_t word = u[w];
    if (!((word >> (j & 31)) & 1u)) return -1;
    int below = __popc(word & own[w] & ((1u << (j & 31)) - 1u));
#pragma unroll 8
    for (int k = 0; k < w; ++k) below += __popc(u[k] & own[k]);
    int64_t byte = (int64_t)(off_s[(br * P + p) * H + h] + below) * entry_bytes;
    if (dst_base) byte += dst_base[br] - (int64_t)off_s[br * PH] * entry_bytes;
    if (capacity >= 0 && byte + entry_bytes > capacity) {
      atomicExch(status, SPARSP_ERR_CAPACITY);  // would overflow: left out
      return -1;
    }
    return byte;
  };
  // Loads the next block into stage st; false: there is none left.
  auto load_next = [&](int st) -> bool {
    while (next < n_blocks) {
      int after = 0;
      if (kFromMask) after = next + n_units;
      else if (lane == 0) after = n_units + atomicAdd(n_taken, 1);
      for (int full_words = 32; full_words == 32; word += full_words)  // words whose blocks have lower numbers
        full_words = __popc(__ballot_sync(0xffffffffu, word + lane < n_words && pos_s[word + lane + 1] <= next));
      uint32_t left = live_s[word];
      for (int skip = next - pos_s[word]; skip > 0; --skip) left &= left - 1u;
      const int bit = __ffs(left) - 1, bh = word / Wd, w = word - bh * Wd, j = w * 32 + bit;
      // its owner, looked for by a lane per rank
      int p = __ffs(__ballot_sync(0xffffffffu, lane < P && ((own_s[lane * Wd + w] >> bit) & 1u))) - 1;
      if (p < 0)
        p = 31 + __ffs(__ballot_sync(0xffffffffu, lane + 32 < P && ((own_s[(lane + 32) * Wd + w] >> bit) & 1u)));
      const int bb = bh / H, h = bh - bb * H;
      bool any = false;
#pragma unroll 1
      for (int r = lane; r < P; r += 32) {
        const int64_t d = destination(bb, h, j, p, r);
        dst_s[st][r] = d;
        any = any || d >= 0;
      }
      next = __shfl_sync(0xffffffffu, after, 0);
      if (!__any_sync(0xffffffffu, any)) continue;  // (no room for any of its copies)
      if (lane == 0) {
        unsigned char* buf = ring + (size_t)st * entry_bytes;
        ptx::mbar_expect_tx(full + st, 2 * tile_bytes);
        ptx::tma_load_4d(buf, &tmK, full + st, 0, j * b, h, bb);
        ptx::tma_load_4d(buf + tile_bytes, &tmV, full + st, 0, j * b, h, bb);
      }
      return true;
    }
    return false;
  };
  int n = 0;  // blocks loaded
  bool more = true;
  for (int q = 1 - kGatherStages; q < 0 || q < n; ++q) {
    if (q >= 0) {
      const int st = q % kGatherStages;
      const unsigned char* buf = ring + (size_t)st * entry_bytes;
      ptx::mbar_wait_bounded(full + st, (uint32_t)((q / kGatherStages) & 1), &s_abort, status, 50, 200000000LL);
      // (an entry is the K tile and the V tile behind it, here as there)
      for (int r = lane; r < P; r += 32) {
        const int64_t d = dst_s[st][r];
        if (d >= 0) bulk_store(packed + d, buf, (uint32_t)entry_bytes);
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    if (more) {
      // the stage of block q - 1 may be refilled once every lane's stores have read it
      asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
      __syncwarp();
      more = load_next(n % kGatherStages);
      n += more ? 1 : 0;
    }
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

int launch_demand_pack(const sparsp_shape& s, const Geometry& g, const uint32_t* mask, const int32_t* rank, int P,
                       int flags, const void* K, const void* V, uint32_t* U, int32_t* cnt, int64_t* seg_off,
                       int64_t* seg_total, int64_t* volume, void* packed, int64_t capacity, const int64_t* dst_base,
                       char* ws, const WsLayout& L, cudaStream_t st) {
  int rc = check_consumers(g, P);
  if (rc != SPARSP_OK) return rc;
  const int local = (flags & SPARSP_INCLUDE_LOCAL) ? 1 : 0;
  int32_t* status = (int32_t*)(ws + L.status);
  const int64_t T = (int64_t)g.B * P * P * g.H, tile_bytes = 2LL * g.b * g.d;
  const int n_copy = pack_warps((int)tile_bytes);
  const int64_t n_words = (int64_t)g.B * g.H * g.Wd;
  int64_t smem = n_copy * kGatherStages * 2 * tile_bytes + (T + 1 + 2 * n_words + 1 + (int64_t)P * g.Wd) * 4;
  const int64_t n_mask = n_words * g.NB, blocks = (int64_t)g.B * g.H * g.NB, a_block_a_warp = 148 * n_copy;
  const bool from_mask = n_mask <= (blocks <= kFromMaskFew * a_block_a_warp ? kMaskMax : kMaskMaxMany) &&
                         blocks <= kFromMaskBlocks * a_block_a_warp &&
                         smem + n_words * P * 4 <= kGatherSmem;
  PackLaunch c;
  if (T <= kScanMax && smem <= kGatherSmem) {
    auto kern = from_mask ? gather_kernel<true> : gather_kernel<false>;
    if (from_mask) smem += n_words * P * 4;
    if ((rc = prepare_pack(s, g, K, V, (const void*)kern, (int)smem, &c)) != SPARSP_OK) return rc;
    int32_t* n_taken = (int32_t*)(ws + L.n_entries);  // zeroed by the union's launch
    if (!from_mask) SPARSP_CUDA_OK(launch_union(g, mask, rank, P, local, U, cnt, nullptr, n_taken, st));
    SPARSP_CUDA_OK(launch_kernel(kern, c.grid, kGatherThreads, (size_t)smem, st, c.tk, c.tv, mask, U, rank, cnt, g.B,
                                 g.H, g.NB, g.Wd, P, local, g.b, c.tile_bytes, n_copy, seg_off, seg_total, volume,
                                 dst_base, capacity, (unsigned char*)packed, n_taken, status));
    return SPARSP_OK;
  }
  const int ring = n_copy * kPackStages * (int)tile_bytes;
  if ((rc = prepare_pack(s, g, K, V, (const void*)pack_kernel, ring, &c)) != SPARSP_OK) return rc;
  int64_t* dst = dst_table(ws, L);
  int32_t* src = src_list(ws, L, g, P);
  int32_t* n_src = (int32_t*)(ws + L.n_entries);
  SPARSP_CUDA_OK(launch_plan(g, mask, rank, P, local, U, cnt, seg_off, seg_total, volume, dst_base, capacity, dst, src,
                             n_src, received_table(ws, L, g, P), status, st));
  SPARSP_CUDA_OK(launch_kernel(pack_kernel, c.grid, 32 * n_copy, (size_t)ring, st, c.tk, c.tv, dst, P, src, n_src, g.H,
                               g.NB, g.b, c.tile_bytes, (unsigned char*)packed, status));
  return SPARSP_OK;
}

// ------------------------------------------------------------------------------------------------
// Pack of ONE (consumer, producer) segment (Section 6.1: the producer packs the payload of one consumer into the slot
// designated for that pair).  Entry (h, j) sits where it sits inside the consumer's buffer, minus the segment's first
// entry, so that consumer and producer derive the same byte ranges from the demand counts.
// The entries are U[consumer][h] & own[producer], head by head, blocks ascending.  Their places in the slot are
// consecutive, so a warp that takes every n-th entry finds its head in the offsets and its block by counting bits: no
// tables and no launch that fills them.  Tiles move as in pack_kernel.  HBM-bound: seven segments of 175 MB, read and
// written, 426 us with tables, 382-384 this way (6.4 TB/s); 421 with a run of consecutive entries per warp instead of
// every n-th.  Three tiles per warp: with two loads in flight reads and writes alternate best (four 390, five 394).
// Small segments, 80 entries of 40 heads / 400 of 200: 9.2 / 9.0 us with tables, 6.2 / 6.2; walking from head to head
// 18 / 52.
// ------------------------------------------------------------------------------------------------
constexpr int kSegmentStages = 3;

__global__ void __launch_bounds__(32 * kPackMaxWarps)
    segment_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                   const uint32_t* __restrict__ U, const int32_t* __restrict__ rank, int H, int NB, int Wd, int P,
                   int consumer, int producer, const int64_t* __restrict__ seg_off, const int32_t* __restrict__ cnt,
                   int b, uint32_t tile_bytes, unsigned char* __restrict__ slot, int64_t capacity,
                   int32_t* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ uint64_t full_all[kPackMaxWarps * kSegmentStages];
  __shared__ int s_abort;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
  uint64_t* full = full_all + warp * kSegmentStages;
  unsigned char* ring = smem_raw + (size_t)warp * kSegmentStages * tile_bytes;  // this warp's buffers
  if (threadIdx.x == 0) s_abort = 0;
  if (lane == 0) {
    for (int st = 0; st < kSegmentStages; ++st) ptx::mbar_init(full + st, 1);
    ptx::mbar_init_fence();
  }
  enter_grid(U, rank, seg_off, cnt);
  __syncthreads();
  uint32_t own = 0;  // blocks of the producer, a word per lane
#pragma unroll 8
  for (int w = 0; w < Wd; ++w) {
    const int j = w * 32 + lane;
    const uint32_t word = __ballot_sync(0xffffffffu, (j < NB ? rank[j] : ~producer) == producer);
    if (lane == w) own = word;
  }
  const int64_t* off = seg_off + ((int64_t)consumer * P + producer) * H;  // batch item 0
  const int64_t first = off[0];
  const int n_entries = (int)(off[H - 1] + cnt[((int64_t)consumer * P + producer) * H + H - 1] - first);
  const int unit = blockIdx.x * n_warps + warp, n_units = gridDim.x * n_warps;
  // Every second consumer's entries are walked backwards: the tiles that were read last for one consumer are the first
  // ones for the next and still in L2.
  const bool back = consumer & 1;
  int n_local = n_entries > unit ? 2 * ((n_entries - unit + n_units - 1) / n_units) : 0;  // K (even) or V (odd) tiles
  auto entry = [&](int q) { return back ? n_entries - 1 - unit - (q >> 1) * n_units : unit + (q >> 1) * n_units; };
  if (n_local > 0) {
    const uint32_t* u_row = U + (int64_t)consumer * H * Wd;
    // the head that entry e belongs to, the last one that begins at or before it
    auto head_of = [&](int e) -> int {
      int lo = 0, end = H;
      while (end - lo > 1) {
        const int step = (end - lo + 31) / 32, h = lo + lane * step;
        const int c = __popc(__ballot_sync(0xffffffffu, h < end && off[h] - first <= e));
        lo += max(c - 1, 0) * step;
        end = min(end, lo + step);
      }
      return lo;
    };
    auto head_words = [&](int h) { return lane < Wd ? u_row[(int64_t)h * Wd + lane] & own : 0u; };
    // The head of the next entry to load, its first entry, and its words on their way.  Where the heads begin is kept a
    // lane per head, 32 of them in the direction of the walk, so that a look needs no load.
    int h, at, h0, x_at;
    uint32_t words;
    auto keep_heads = [&](int from) {
      h0 = from;
      const int x = back ? h0 - lane : h0 + lane;
      x_at = x >= 0 && x < H ? (int)(off[x] - first) : back ? 0 : INT_MAX;
    };
    auto look_up = [&](int e) {
      uint32_t begun = __ballot_sync(0xffffffffu, x_at <= e);  // of the heads kept: from one on (back), or up to one
      if (begun == (back ? 0u : ~0u)) {
        keep_heads(head_of(e));
        begun = __ballot_sync(0xffffffffu, x_at <= e);
      }
      const int found = back ? __ffs(begun) - 1 : __popc(begun) - 1;
      h = back ? h0 - found : h0 + found;
      at = __shfl_sync(0xffffffffu, x_at, found);
      words = head_words(h);
    };
    keep_heads(head_of(entry(0)));
    look_up(entry(0));
    // head * NB + block of entry e, which has been looked up; -1 where there is none, should the counts promise more
    // than there are
    auto block_of = [&](int e) -> int {
      int total;
      const int below = bits_below(words, lane, &total), k = e - at;
      if (k >= total) return -1;
      const int w = 31 - __clz(__ballot_sync(0xffffffffu, words != 0u && below <= k));
      uint32_t left = __shfl_sync(0xffffffffu, words, w);
      for (int skip = k - __shfl_sync(0xffffffffu, below, w); skip > 0; --skip) left &= left - 1u;
      return h * NB + w * 32 + __ffs(left) - 1;
    };
    int s_load = 0;
    auto issue_load = [&](int q) {
      if ((q & 1) == 0) s_load = block_of(entry(q));
      if (s_load < 0) {
        n_local = q;
        return;
      }
      if (lane == 0) {
        uint64_t* bar = full + q % kSegmentStages;
        const int hd = s_load / NB;
        ptx::mbar_expect_tx(bar, tile_bytes);
        ptx::tma_load_4d(ring + (size_t)(q % kSegmentStages) * tile_bytes, q & 1 ? &tmV : &tmK, bar, 0, (s_load - hd * NB) * b,
                         hd, 0);
      }
      if ((q & 1) && q + 1 < n_local) look_up(entry(q + 1));
    };
    for (int q = 0; q < kSegmentStages - 1 && q < n_local; ++q) issue_load(q);
    for (int q = 0; q < n_local; ++q) {
      const int64_t e = entry(q);
      ptx::mbar_wait_bounded(full + q % kSegmentStages, (uint32_t)((q / kSegmentStages) & 1), &s_abort, status, 50,
                             200000000LL);
      if (lane == 0) {
        if ((e + 1) * 2 * tile_bytes <= capacity)
          bulk_store(slot + (2 * e + (q & 1)) * tile_bytes, ring + (size_t)(q % kSegmentStages) * tile_bytes, tile_bytes);
        else
          atomicExch(status, SPARSP_ERR_CAPACITY);  // does not fit: left out
      }
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      if (q + kSegmentStages - 1 < n_local) {
        // the buffer of item q - 1 may be refilled once its store has read it
        asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
        __syncwarp();
        issue_load(q + kSegmentStages - 1);
      }
    }
  }
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

int launch_pack_segment(const sparsp_shape& s, const Geometry& g, const uint32_t* U, const int32_t* rank, int P,
                        int consumer, int producer, const int64_t* seg_off, const int32_t* cnt, const void* K,
                        const void* V, void* dst, int64_t capacity, char* ws, const WsLayout& L, cudaStream_t st) {
  PackLaunch c;
  const int n_warps = pack_warps(g.b * g.d * 2), smem = n_warps * kSegmentStages * g.b * g.d * 2;
  const int rc = prepare_pack(s, g, K, V, (const void*)segment_kernel, smem, &c);
  if (rc != SPARSP_OK) return rc;
  SPARSP_CUDA_OK(launch_kernel(segment_kernel, c.grid, 32 * n_warps, (size_t)smem, st, c.tk, c.tv, U, rank, g.H, g.NB, g.Wd, P,
                               consumer, producer, seg_off, cnt, g.b, c.tile_bytes, (unsigned char*)dst, capacity,
                               (int32_t*)(ws + L.status)));
  return SPARSP_OK;
}

// ------------------------------------------------------------------------------------------------
// Allocation-free planning call: the same two launches, which need no scratch when no destinations are asked for, so a
// caller that cannot allocate device memory at all can still obtain unions, counts, offsets and volumes.
// ------------------------------------------------------------------------------------------------
constexpr int kPlanMaxRanks = 64;         // n_ranks limit of the allocation-free call
constexpr int kPlanMaxBatchRanks = 1024;  // batch * n_ranks limit

}  // namespace sparsp

using namespace sparsp;

extern "C" SPARSP_API int sparsp_demand_plan_noalloc(const sparsp_shape* shape, const uint32_t* mask,
                                                     const int32_t* rank_of_block, int32_t n_ranks,
                                                     int32_t flags, uint32_t* union_mask, int32_t* cnt,
                                                     int64_t* seg_offset, int64_t* seg_total,
                                                     int64_t* volume_bytes, void* stream) {
  Geometry g;
  int rc = make_geometry(shape, &g);
  if (rc != SPARSP_OK) return rc;
  if (n_ranks < 1 || n_ranks > kPlanMaxRanks || (int64_t)g.B * n_ranks > kPlanMaxBatchRanks) {
    set_error("sparsp_demand_plan_noalloc supports n_ranks <= %d and batch * n_ranks <= %d (got %d, %lld)",
              kPlanMaxRanks, kPlanMaxBatchRanks, n_ranks, (long long)g.B * n_ranks);
    return SPARSP_ERR_CAPACITY;
  }
  if (flags & ~SPARSP_INCLUDE_LOCAL) {
    set_error("sparsp_demand_plan_noalloc accepts only SPARSP_INCLUDE_LOCAL (got 0x%x)", flags);
    return SPARSP_ERR_INVALID_ARG;
  }
  if (!mask || !rank_of_block || !union_mask || !cnt || !seg_offset || !seg_total || !volume_bytes) {
    set_error("sparsp_demand_plan_noalloc: NULL argument");
    return SPARSP_ERR_INVALID_ARG;
  }
  if ((uintptr_t)seg_offset % 8 || (uintptr_t)seg_total % 8 || (uintptr_t)volume_bytes % 8 ||
      (uintptr_t)mask % 4 || (uintptr_t)union_mask % 4 || (uintptr_t)cnt % 4 || (uintptr_t)rank_of_block % 4) {
    set_error("sparsp_demand_plan_noalloc: misaligned argument");
    return SPARSP_ERR_INVALID_ARG;
  }
  SPARSP_CUDA_OK(launch_plan(g, mask, rank_of_block, n_ranks, (flags & SPARSP_INCLUDE_LOCAL) ? 1 : 0, union_mask, cnt,
                             seg_offset, seg_total, volume_bytes, nullptr, -1, nullptr, nullptr, nullptr, nullptr,
                             nullptr, (cudaStream_t)stream));
  return SPARSP_OK;
}
