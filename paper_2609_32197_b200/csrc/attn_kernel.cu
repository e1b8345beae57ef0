// Step 3: block-sparse FlashAttention forward on tcgen05 tensor cores (sm_100a).
//
// Work item = ONE 128-row Q tile of one (batch, head) with one fp32 accumulator O in tensor memory:
//   block = 128: the Q tile is one query block; the item walks that block's kept KV blocks.
//   block = 64 : two query blocks (chosen by a pairing pass so that their kept lists overlap) are stacked into the Q
//                tile (full-rate M = 128 MMAs); a KV tile is two entries of the UNION of their kept lists (128 keys,
//                full-rate N = 128); each 64x64 quadrant the mask does not keep is zeroed in P.
// The kernel is persistent: one CTA per SM takes items from a global counter (or in turn, see Source); the next item's
// kept list, Q tile and first K/V tiles overlap the current item's last tiles, its first Q K^T the epilogue.  Where an
// item ends, only the warpgroup of its last tile waits for the accumulator and writes the rows; the other one is
// already at the next item, whose Q tile has a buffer of its own: the next one of the K ring, which gets the finished
// item's Q buffer in exchange.  (Both warpgroups writing half of the columns, the Q tile behind the last Q K^T in a
// buffer that is always Q's: 13 heads x 2 x 6034 tokens, 9 tiles an item, 86.9 us a call, now 78.2; 16 x 18600 with 6
// to 30 tiles 306 / 282; 40 x 75600, 59 tiles, 10.05 / 9.82 ms; one hop of it over 8 ranks, 2 to 8 tiles, 64.1 / 61.1.
// Tried on top and no better: rows through shared memory and a TMA store, lists for one or two items more, tiles dealt
// so that the warpgroups take turns at writing.)
// Every softmax warpgroup has a buffer of its own for scores S = Q K^T in tensor memory (128 fp32 columns), so that the
// tensor pipe always has the next tiles' MMAs queued while the softmax of the current tile runs.  Tiles are numbered g
// = 0, 1, 2, ...  across the CTA's items; every ring, buffer and barrier phase follows g.
//   d = 128: two warpgroups.  S 2 x 128 columns, P 64 columns of packed bf16, O 128 columns, 16 columns for the row
//            sums.  Q K^T of tile g+2 starts as soon as the scores of tile g have been READ.  A tile moves 160 KB
//            through shared memory (64 KB of TMA writes, 96 KB of operands), 1250 clocks at 128 bytes a clock; ordinary
//            tiles take 1400.
//   d = 64:  three warpgroups.  A tile is half of that and its 16384 exponentials bound it, with two warps a scheduler
//            more by their latencies (1495 clocks) than by the special-function unit (683), so there is a third one.  S
//            3 x 128 columns, P in the place of the scores it was made from, O 64 + 16 columns; Q K^T of tile g+3
//            starts when P V of tile g has read P.  Two warpgroups with P buffers of their own / three: 13 heads x 2 x
//            6034 tokens 78.7 / 76.0 us a call, 48 x 17776 1380 / 1321, 16 x 18600 with threshold lists 282 / 258, 27 x
//            27403 from a packed buffer 279 / 244.
// P V of tile g is issued as soon as P_g is written.
// Warp roles (512 or 640 threads = 4 or 5 warpgroups; the first two hand most of their registers to the others):
//   warp 0      TMA producer of Q (per item) and K, which share a ring of buffers
//   warp 1      issues every Q K^T          warp 2      issues every P V
//   warp 3      TMA producer of the V ring
//   warp 4      builds the kept / union list of the NEXT items (two list buffers)
//   warps 5-7   clear the output rows of query blocks that keep nothing
//   warps 8-    softmax: warpgroup w of kWGs takes the tiles with g % kWGs = w
// (A producer is one thread running a chain of dependent instructions next to busy softmax warps: it gets an
// instruction issued every ~8 cycles, so K and V loads have a warp each and keep per-tile work minimal.)  A softmax
// thread owns one query row of its tile: at d = 128 the whole 128-column row of S sits in registers, at d = 64, with
// fewer registers a thread, 32 columns and the next 32 on their way.  Ordinary items run
// without a row maximum: load scores -> exponentials -> store P, relative to 0 (K / V source) or to the row's maximum
// over the item's first tile (packed source), which the warpgroup of that tile hands to the others; the tensor pipe
// takes the row sums.  Whether that was right is seen from the finished row sums and the exponents on the way, and an
// item that left the range is computed again (kRefZero ... below).  Only such an item, and rows whose first scores are
// out of range, take their maxima as they go: the threads that own the same row (one per warpgroup) then share the
// reference through shared memory and take their decisions strictly in tile order (mbarriers of the row group hand the
// turn from one to the next), and O is rescaled lazily, only when a row's maximum has grown by more than 2^8 since the
// reference last moved.  The thread that decides so waits for every P V issued so far, but only behind its
// exponentials, which need nothing but the new reference: those of neighbouring tiles overlap.  (Waiting and rescaling
// before them, us a call with Q times 40: 5 heads x 492 blocks of 64 x 64, 15 % kept 930, now 632; 9 x 324 of 64 x 128
// 1787 / 1039; 4 x 300 of 128 x 128, 10 % 554 / 363.  16 columns of the accumulator at a time also at d = 128: 24 x
// 24576 from a packed buffer, Q times 60 638, now 578.)  (The range used to be proved beforehand, by Cauchy-Schwarz
// from key norms that a pass over K took ahead of every call and row norms taken from the Q tile of every item, and not
// at all for a packed source, whose tiles all took their maximum in turns.  us per call then and now: one hop of 40
// heads x 75600 over 8 ranks, 7 tiles an item, 97-112 -> 75; 24 x 24576 from one rank's whole buffer 437-445 ->
// 415-425; 13 heads x 2 x 6034 92-101 -> 85-93; all of 40 x 75600 10.1-10.5 -> 9.7-10.2 ms.)
// The block-64 pairing and the order of a head's items (longest list first) come from attn_prep_kernel; calls of few
// items have their CTAs put them in order (kDirect, kPackedDirect below).
// Every mbarrier wait is bounded; a wait that runs out sets SPARSP_ERR_TIMEOUT in the status word
// and raises a CTA-wide flag that makes all later waits fall through, so the CTA still drains.
#include <algorithm>
#include <type_traits>

#include "block_sets.cuh"
#include "common.cuh"
#include "item_queue.cuh"
#include "sm100_ptx.cuh"

namespace sparsp {

using namespace ptx;

struct AttnParams {
  const uint32_t* mask;
  // work items of every (batch, head), [B*H][2*ceil(NB/2)]: block 64: two query blocks per item (the second may be -1);
  // block 128: one.  Only the first n_items[bh] items of a head exist: every one of them keeps at least one KV block.
  const int32_t* pairs;
  const int32_t* n_items;
  // packed source only: slot[bh][j] = entry index of KV block j in
  // the consumer's packed buffer, or -1 if the consumer owns the block; tile_base = index of the
  // consumer's first tile in the packed tensor map (a device scalar)
  const int32_t* slot;
  const int64_t* tile_base;
  const int32_t* rank;  // packed source: owner of every block, and the rank whose rows are computed
  int consumer;
  // kPackedDirect: what slot and tile_base are made of
  int P;
  const uint32_t* U;
  const int64_t *seg_off, *seg_total, *dst_base;
  int64_t tile_bytes;
  __nv_bfloat16* O;
  float* lse;
  int32_t* status;
  int32_t* work_counter;  // items handed out beyond the first one of every CTA; zeroed by the preparatory launch
  int64_t N;
  int64_t sB, sH, sT;
  int BH, H, NB, Wd;
  int in_place;      // O is Q: no row of an item is written before all of them are known to be right
  float scale_log2;  // softmax scale * log2(e)
  long long wait_limit;
};

// register budget per thread after the warpgroups re-balance (d = 128: 256 * 48 + 256 * 208 = 512 * 128; d = 64: 256 *
// 48 + 384 * 128 = 640 * 96, which is what a block of 640 threads is launched with; the softmax warps and the list
// builder spill up to 130 bytes)
#ifndef SPARSP_REGS_UTILITY
#define SPARSP_REGS_UTILITY 48
#define SPARSP_REGS_UTILITY2 48
#define SPARSP_REGS_SOFTMAX 208
#endif
constexpr int kTmemCols = 512;
constexpr int kWorkCounterWord = 8;  // word of the workspace header that holds the attention work counter
constexpr float kGrowThreshold = 8.0f;
// Where an item's softmax rows take the reference that is subtracted from their scores (log2 domain) from:
//   kRefZero   nowhere, it is 0;
//   kRefFirst  the row's maximum over the item's first tile (0 for a row that keeps nothing of it);
//   kRefExact  the row's running maximum, moved lazily and strictly in tile order.
// The first two look at no score behind the first tile, so they are right only for rows whose scores stay near the
// reference.  That is seen at the end of the item: no exponential left the range of normal numbers on the FMA pipe
// (kMaxExponent; the special-function unit saturates to 0 and infinity by itself), the row sum lies within [kMinSum,
// kMaxSum], and no output column ran out of fp32 where the sum is so large that a finite V could do that (above
// kSafeSumZero or kSafeSumFirst; below them it takes |V| > 2^63 or 2^102, and the running maximum allows no more than
// the latter).  Then every term is a normal fp32 and bf16 number of full relative precision, or at most 2^-36 of the
// sum.  An item with a row that fails, one with scores that are no numbers included, is computed again as kRefExact.
// So that this is rare, the four warps of the item's first tile look at it first: rows whose first scores are far from
// 0 take the running maximum from the start, the 32 rows of a warp together (kZeroSample: every eighth score;
// kFirstSample: the maximum that the reference is anyway).  Ordinary scores pass both: with unit-variance Q and K at d
// = 128 they are within +-16.  (us per call of 13 heads x 2 x 6034 tokens, Q times 1, 4 and 60: 87, 144 and 136;
// looking for +-64 only 183 with Q times 4; with range proofs from the norms of rows and keys instead of all this 91,
// 131 and 140.)  All of this follows from the item alone, so a call repeats itself bit for bit whichever CTA takes
// which item.  (A CTA that remembered failures and began its next items further on was right too, but let rows of
// ordinary heads change in their last bit from call to call.)
constexpr int kRefZero = 0, kRefFirst = 1, kRefExact = 2;
constexpr float kMaxExponent = 126.0f;
constexpr float kMinSum = 8.077935669463161e-28f;  // 2^-90
constexpr float kMaxSum = 1.2676506002282294e30f;  // 2^100
constexpr float kSafeSumZero = 1.8446744073709552e19f;  // 2^64
constexpr float kSafeSumFirst = 33554432.0f;            // 2^25: kGrowThreshold and 2^17 keys
constexpr float kZeroSample = 48.0f, kFirstSample = 64.0f;
constexpr int kZeroMinTiles = 4;  // K / V source: shorter items take kRefFirst, whose largest terms are exact
// Tuning switch (compile-time): how many of the exponentials go to the FMA pipe instead of the special-function unit
// (every n-th pair; 0 = none).  The same share everywhere, so that a row's result does not depend on where its tiles
// come from.  us per attention call with every 3rd / 4th / 6th pair:
//   d = 64                   48 heads x 17776 tokens 1393 / 1410 / 1429 (none 1488, every 2nd 3 % slower than every
//                            3rd)
//   d = 128, 64-token blocks 24 x 24576, half of the blocks kept, neighbours alike 3094 / 3219 / -, 8 x 16384 with all
//                            kept 912 / 948 / -, 24 x 24576 with threshold lists 671 / 665 / 681
//   ... 128-token blocks     under the power cap a smaller share is up to 1 % faster: 40 x 75600, 10 % kept 9884 / 9816
//                            / 9903 (none 10596), one hop of it over 8 ranks 60.8 / - / 60.2
#ifndef SPARSP_TUNE_POLY
#define SPARSP_TUNE_POLY 3
#endif

// Lists that the list builder keeps: the current item's and the next one's.  (With 3 or 4 a CTA takes items that one
// with nothing left to do cannot take any more: 9 heads x 10602 tokens 60.8 us a call, 62.2 with 3, 63.2 with 4.)
constexpr int kLists = 2;
// One list entry: a KV block and which of the item's two query blocks keep it (64-token blocks); for a packed source
// the tile index of a remote block in its place.  (A word, or half of one, for both of a tile's entries: with the
// block, the valid keys per query block and the slot in three arrays 48 heads x 17776 took 2 % longer.)
template <bool kPacked>
struct Entry;
template <>
struct Entry<false> {
  using type = uint16_t;
  static constexpr int kFlagShift = 14;  // bits 14, 15: kept by the first, the second query block
};
template <>
struct Entry<true> {
  using type = uint32_t;
  static constexpr int kFlagShift = 30;
  // bits 0-28 are the block's K tile in the packed buffer (its V tile is next)
  static constexpr uint32_t kRemote = 1u << 29;
  static constexpr uint32_t kValue = kRemote - 1u;
};
// Item header, one load for each role: x = batch * H + head; y = entries | kHead... flags (0: there are no more items);
// z = query blocks, first | second << 16 (0xffff: none); w = batch.
constexpr int kHeadEntries = 0xffff, kHeadRagged = 1 << 16, kHeadRefShift = 17, kHeadNoneShift = 19;
// ... and whether all softmax warps meet before the item's rows are written (`placed`), with the parity of that
// meeting.
constexpr int kHeadMeet = 1 << 21, kHeadMeetParityShift = 22;

// Where items and their K / V tiles come from.
//   kQueue         a queue of items made by the preparatory launch, the sequence's own K and V
//   kDirect        the same K and V, but every query block is an item (64-token blocks: not stacked), of which there
//                  are so few that the CTAs take them in turn, in order if there are more of them than CTAs
//   kPacked        a queue of the consumer's items, a packed buffer and the consumer's own K and V
//   kPackedDirect  the same tiles, but the CTAs number the consumer's items and places in the buffer for themselves,
//                  and put the items in order if there are more of them than CTAs
enum class Source { kQueue, kDirect, kPacked, kPackedDirect };

constexpr int kMaxDirect = 2 * 148, kMaxPackedDirect = 1024;  // items of a call without a queue
constexpr int kPackedDirectBlocks = 512;  // blocks of a head up to which that many

template <int D, int BLK>
struct AttnCfg {
  static constexpr bool kStacked = (BLK == 64);  // Q tile = two 64-token query blocks
  static constexpr int kEPT = 128 / BLK;         // kept-list entries per 128-key KV tile
  static constexpr int kStagesK = (D == 64) ? 4 : 3;
  static constexpr int kStagesV = (D == 64) ? 4 : 2;
  static constexpr int kTileBytes = 128 * D * 2;  // one K or V tile
  // Q tile and K ring share kStagesK + 1 buffers: an item's Q tile takes the next buffer of the ring for as long as the
  // item lasts, the buffer of the item before it joins the ring behind (QKRing).
  static constexpr int kBufsQK = kStagesK + 1;
  static constexpr int kOffQK = 0;
  static constexpr int kOffV = kOffQK + kBufsQK * kTileBytes;
  // d = 64 leaves room in tensor memory for 16 more accumulator columns: P V then runs with N = 80, its B
  // operand continuing, 64 columns on, into a constant [128 keys][column 64 = 1, the rest 0] block in shared
  // memory, so that accumulator column 64 is the row sum of P -- taken by the tensor pipe from the very
  // bf16 values it multiplies with V, instead of one more packed add per pair of scores in the softmax warps
  static constexpr bool kOnes = (D == 64);
  static constexpr int kAccCols = D + (kOnes ? 16 : 0);
  // d = 128: the row sum also comes from the tensor pipe, through a separate N = 16 MMA per 16
  // keys against a [16 keys][column 0 = 1] block (2 KB, 128-byte swizzle like a V box), into 16 tensor-memory columns
  // of its own -- which exist only if P keeps ONE buffer instead of two (tensor memory is full otherwise)
  static constexpr bool kSum128 = (D == 128);
  // Softmax warpgroups, each of which takes every kWGs-th tile and has an S buffer.  Three: P takes the place of the
  // scores it was made from.  Two: one P buffer for both.
  static constexpr int kWGs = D == 64 ? 3 : 2;
  static constexpr bool kInPlaceP = kWGs == 3;
  static constexpr int kThreads = (2 + kWGs) * 128;  // two warpgroups of utility warps before them
  static constexpr int kRegsSoftmax = kWGs == 3 ? 128 : SPARSP_REGS_SOFTMAX;
  static constexpr int kListReaders = 4 + 4 * kWGs;  // two producers, two issuers, the softmax warps
  static constexpr int kOffOnes = kOffV + kStagesV * kTileBytes;  // bf16 [128][64], 128-byte swizzle like a V box
  static constexpr int kOffEnt = kOffOnes + (kOnes ? 128 * 128 : 2048);  // entries [kLists][1024]
  static constexpr int kOffRef = kOffEnt + kLists * kMaxBlocks * 4;  // float [4 items][128] reference per row
  static constexpr int kOffBars = kOffRef + 4 * 128 * 4;
  static constexpr int kNumBars = 2 * (kBufsQK + kStagesV) + 3 * kWGs + 4 + 1 + 2 * kLists + 4 + 8 * kWGs + 1;
  static constexpr int kColS = 0;    // S buffers: 128 columns each
  static constexpr int kColP = 256;  // d = 128: P in columns [256, 320), row sums in [320, 336)
  static constexpr int kColO = 384;  // accumulator: columns [384, 384 + d)
  static constexpr int kColL = kOnes ? kColO + D : 320;  // row sums (column 0 of 16), where the tensor pipe takes them
  static constexpr int kOffHead = (kOffBars + 8 * kNumBars + 15) / 16 * 16;  // int4 [kLists]
  static constexpr int kOffMisc = kOffHead + 16 * kLists;
  static constexpr int kTotal = kOffMisc + 64;
  static constexpr int kDynamic = kTotal + 1024;  // slack for the 1024-byte alignment of the base
  // kPackedDirect: uint32 own[P][Wd], int32 first[P][Wd] (places of a head's blocks), uint32 union[32], uint8
  // rank[1024]
  static constexpr int kOffOwn = kTotal, kOffFirst = kOffOwn + kMaxRanks * kMaxWords * 4;
  static constexpr int kOffUnion = kOffFirst + kMaxRanks * kMaxWords * 4, kOffRank = kOffUnion + kMaxWords * 4;
  static constexpr int kOffPackedOrder = kOffRank + kMaxBlocks;  // uint16 items in order
  static constexpr int kDynamicDirect = kOffPackedOrder + 2 * kMaxPackedDirect + 1024;
  // (while items are put in order, the places of entries and `first` hold counts and the list of own blocks)
  static_assert(4 * (kMaxBlocks + 1) <= kLists * kMaxBlocks * 4, "room for the counts");
  static_assert(2 * kMaxBlocks <= kMaxRanks * kMaxWords * 4, "room for the list");
  // kDirect: the same lengths, uint16 items in order
  static constexpr int kOffLength = kTotal, kOffOrder = kOffLength + 4 * kMaxDirect;
  static_assert(kDynamicDirect <= 232448, "shared memory budget");
};

// Packed fp32 pairs (one instruction for two lanes' worth of fused multiply-add / add).
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  unsigned long long ra, rb, rc, rd;
  float2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rc) : "f"(c.x), "f"(c.y));
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(rd) : "l"(ra), "l"(rb), "l"(rc));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
  return d;
}
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) {
  unsigned long long ra, rb, rd;
  float2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(ra) : "f"(a.x), "f"(a.y));
  asm("mov.b64 %0, {%1, %2};" : "=l"(rb) : "f"(b.x), "f"(b.y));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(rd) : "l"(ra), "l"(rb));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(rd));
  return d;
}

// max(|a|, |b|, |c|), not a number if any of them is none.
__device__ __forceinline__ float max_abs3(float a, float b, float c) {
  float d;
  asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// The larger of the two, not a number if one of them is none.
__device__ __forceinline__ float max_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}

// 2^x for a pair of fp32 values on the FMA/ALU pipes (no special-function unit): round-to-nearest
// split x = i + f, f in [-0.5, 0.5], cubic minimax polynomial for 2^f (relative error 7.5e-5, far
// below bf16 rounding), exponent added into the bit pattern.  The result is right for |i| <= 126, and infinite in bf16
// where x is not a number.  kTrack: *i_max collects the largest |i|.  kClamp: x is clamped at -126 first (result >=
// 2^-126).
template <bool kClamp, bool kTrack>
__device__ __forceinline__ float2 exp2_poly2(float2 x, float* i_max) {
  const float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds to an integer in the low mantissa bits
  if (kClamp) {
    x.x = max_nan(x.x, -126.0f);
    x.y = max_nan(x.y, -126.0f);
  }
  const float2 t = fadd2(x, make_float2(kMagic, kMagic));
  const float2 fi = fadd2(t, make_float2(-kMagic, -kMagic));
  if (kTrack) *i_max = max_abs3(fi.x, fi.y, *i_max);
  const float2 f = fadd2(x, make_float2(-fi.x, -fi.y));
  float2 q = ffma2(f, make_float2(0.0551716685f, 0.0551716685f), make_float2(0.2426111251f, 0.2426111251f));
  q = ffma2(q, f, make_float2(0.6932609677f, 0.6932609677f));
  q = ffma2(q, f, make_float2(0.9999280572f, 0.9999280572f));
  q.x = __int_as_float(__float_as_int(q.x) + (__float_as_int(t.x) << 23));
  q.y = __int_as_float(__float_as_int(q.y) + (__float_as_int(t.y) << 23));
  return q;
}

// The output rows of query block i: zeros and a log-sum-exp of -inf.  One warp, 32 bytes a lane where the layout
// allows.
template <int D, int BLK>
__device__ __forceinline__ void clear_rows(const AttnParams& p, int bh, int i) {
  const int lane = threadIdx.x & 31;
  const int64_t tok0 = (int64_t)i * BLK;
  const int n = (int)min((int64_t)BLK, p.N - tok0);
  __nv_bfloat16* o = p.O + (bh / p.H) * p.sB + (bh % p.H) * p.sH + tok0 * p.sT;
  if (((reinterpret_cast<uintptr_t>(o) | (uintptr_t)(p.sT * 2)) & 31) == 0) {
    constexpr int LPT = D / 16;  // lanes per row
    o += (lane / LPT) * p.sT + (lane % LPT) * 16;
#pragma unroll 8
    for (int r = lane / LPT; r < n; r += 32 / LPT, o += (32 / LPT) * p.sT)
      asm volatile("st.global.v8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"l"(o), "r"(0) : "memory");
  } else {
    constexpr int LPT = D / 8;
    o += (lane / LPT) * p.sT + (lane % LPT) * 8;
#pragma unroll 8
    for (int r = lane / LPT; r < n; r += 32 / LPT, o += (32 / LPT) * p.sT)
      *reinterpret_cast<uint4*>(o) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (p.lse)
    for (int r = lane; r < n; r += 32) p.lse[bh * p.N + tok0 + r] = -INFINITY;
}

template <int D, int BLK, Source kSource>
__global__ void __launch_bounds__(AttnCfg<D, BLK>::kThreads, 1)
    attn_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmP,
                    const AttnParams p) {
  using C = AttnCfg<D, BLK>;
  constexpr bool kDirect = kSource == Source::kDirect, kPackedDirect = kSource == Source::kPackedDirect;
  constexpr bool kPacked = kSource == Source::kPacked || kPackedDirect;
  constexpr int SV = C::kStagesV;
  extern __shared__ unsigned char smem_dyn[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_dyn) + 1023) & ~uintptr_t(1023));
  unsigned char* sQK = smem + C::kOffQK;
  unsigned char* sV = smem + C::kOffV;
  using E = Entry<kPacked>;
  using EntT = typename E::type;
  EntT* sEnt = reinterpret_cast<EntT*>(smem + C::kOffEnt);  // [kLists][kMaxBlocks]
  volatile float* sRef = reinterpret_cast<volatile float*>(smem + C::kOffRef);  // [4][128]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::kOffBars);
  uint64_t* qk_full = bars;                  // a Q or K tile has landed
  uint64_t* qk_empty = qk_full + C::kBufsQK;  // ... and every Q K^T that reads it has completed
  uint64_t* v_full = qk_empty + C::kBufsQK;
  uint64_t* v_empty = v_full + SV;
  uint64_t* s_full = v_empty + SV;  // [kWGs] S buffer written by a Q K^T
  // [kWGs] S buffer read into registers by its 4 softmax warps (not where P takes its place)
  uint64_t* s_free = s_full + C::kWGs;
  uint64_t* p_full = s_free + C::kWGs;  // [kWGs] P of a tile written by its 4 softmax warps
  // [4] the P V of tile g arrives on o_full[g % 4].  Four barriers, because a parity wait can only tell the phase a
  // barrier is in from the one before.  d = 128: a softmax thread that wants P V g-1 has itself seen P V g-3 complete,
  // and P V g+2 cannot complete before that thread has stored P_g.  d = 64: P V g-3 was complete when the Q K^T whose
  // scores it holds was issued.
  uint64_t* o_full = p_full + C::kWGs;
  uint64_t* o_drained = o_full + 4;      // the item's accumulator has been read out by the four warps that write it
  uint64_t* list_ready = o_drained + 1;  // [kLists] list buffer filled
  uint64_t* list_free = list_ready + kLists;  // [kLists] list buffer no longer needed by its kListReaders
  // [4] the four warps that own an item's first tile have left what it says in s_exact and, if that is the reference,
  // in sRef.  Four, because a warpgroup that waits for it may be up to three tiles and as many items behind.
  uint64_t* ref_ready = list_free + kLists;
  // [2][kWGs][4] the warpgroup's warp of a row group has decided about the running maximum of a tile.  Two in turn,
  // because it may decide about the first tile of the next item before the warp behind it has noticed.  (Not named
  // barriers, which cannot be bounded: after a wait that has run out two warps need not agree on who takes turns.
  // Every lane arrives: with one lane behind a __syncwarp and the count of waits in shared memory 13 heads x 2 x 6034,
  // Q times 8, took 138 us, not 132.)
  uint64_t* turn = ref_ready + 4;
  // All softmax warps have come to the end of an item that they meet at.  In-place calls: all items, so that it is
  // known whether the item is to be computed again.  Else: items that are computed again, so that the rows of the first
  // pass, which another warpgroup may have written, and written behind its arrival on list_free, come before those of
  // the second.
  uint64_t* placed = turn + 8 * C::kWGs;
  int4* s_head = reinterpret_cast<int4*>(smem + C::kOffHead);  // [kLists] item headers
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + C::kOffMisc + 4);
  // [4 items][4 row groups] the group's rows take the running maximum
  volatile uint8_t* s_exact = reinterpret_cast<volatile uint8_t*>(smem + C::kOffMisc + 16);
  // [kLists] the item is to be computed again
  volatile int* s_failed = reinterpret_cast<volatile int*>(smem + C::kOffMisc + 32);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // ---- setup ------------------------------------------------------------------------------
  if (tid == 0) {
    prefetch_tmap(&tmQ);
    prefetch_tmap(&tmK);
    prefetch_tmap(&tmV);
    for (int s = 0; s < C::kBufsQK; ++s) {
      mbar_init(qk_full + s, 1);
      mbar_init(qk_empty + s, 1);
    }
    for (int s = 0; s < SV; ++s) {
      mbar_init(v_full + s, 1);
      mbar_init(v_empty + s, 1);
    }
    for (int s = 0; s < C::kWGs; ++s) {
      mbar_init(s_full + s, 1);
      mbar_init(s_free + s, 4);
      mbar_init(p_full + s, 4);
    }
    for (int s = 0; s < kLists; ++s) {
      mbar_init(list_ready + s, 1);
      mbar_init(list_free + s, C::kListReaders);
    }
    for (int s = 0; s < 4; ++s) mbar_init(o_full + s, 1);
    mbar_init(o_drained, 4);
    for (int s = 0; s < 4; ++s) mbar_init(ref_ready + s, 4);
    for (int s = 0; s < 8 * C::kWGs; ++s) mbar_init(turn + s, 32);
    mbar_init(placed, 4 * C::kWGs);
    mbar_init_fence();
    *s_abort = 0;
  }
  {
    // key row r holds column 64 + c at byte r*128 + ((c/8 ^ (r & 7)) << 4) + (c%8)*2 (the swizzle of a TMA box);
    // 128 key rows at d = 64 (one block for a whole tile), 16 at d = 128 (every group of 16 keys uses the same)
    uint4* ones = reinterpret_cast<uint4*>(smem + C::kOffOnes);
    for (int idx = tid; idx < (C::kOnes ? 128 : 16) * 8; idx += C::kThreads) {
      const int r = idx >> 3, chunk = idx & 7;
      ones[idx] = make_uint4(chunk == (r & 7) ? 0x3F80u : 0u, 0u, 0u, 0u);  // bf16 1.0 in element 0 of logical chunk 0
    }
    fence_proxy_async_smem();  // read by the tensor pipe
  }
  if (warp == 1) {
    tmem_alloc(s_tmem, kTmemCols);
    tmem_relinquish();
  }
  enter_grid();  // (barriers, tensor memory and constants are set up while the launch before still runs)
  uint32_t* sOwn = reinterpret_cast<uint32_t*>(smem + C::kOffOwn);
  uint8_t* sRank = smem + C::kOffRank;
  uint32_t* sLength = reinterpret_cast<uint32_t*>(smem + C::kOffLength);
  uint16_t* sOrder = reinterpret_cast<uint16_t*>(smem + (kPackedDirect ? C::kOffPackedOrder : C::kOffOrder));
  if constexpr (kDirect) {
    // More items than CTAs: every CTA puts all of them in order, the longest list first.  A mask row is an item; short
    // rows share a warp's load.
    const int n = p.BH * p.NB;
    if (n > (int)gridDim.x) {
      int width = 1;  // lanes per row: the next power of two
      while (width < p.Wd) width <<= 1;
      const int per_warp = 32 / width, w = lane & (width - 1);
      constexpr int kFlight = 4, kWarps = C::kThreads / 32;
      for (int first = warp * per_warp; first < n; first += kFlight * kWarps * per_warp) {  // (the same for all lanes)
        const int row0 = first + lane / width;
        uint32_t v[kFlight];
#pragma unroll
        for (int u = 0; u < kFlight; ++u) {
          const int row = row0 + u * kWarps * per_warp;
          v[u] = row < n && w < p.Wd ? p.mask[(int64_t)row * p.Wd + w] : 0u;
        }
#pragma unroll
        for (int u = 0; u < kFlight; ++u) {
          const int row = row0 + u * kWarps * per_warp;
          int len = __popc(v[u]);
          for (int s = 1; s < width; s <<= 1) len += __shfl_xor_sync(0xffffffffu, len, s);
          if (w == 0 && row < n) sLength[row] = (uint32_t)len << 16 | (uint32_t)(0xffff - row);
        }
      }
      if (tid < 4 && n + tid < ((n + 3) & ~3)) sLength[n + tid] = 0u;
      __syncthreads();
      for (int t = tid; t < n; t += C::kThreads) {
        const uint32_t key = sLength[t];
        int place = 0;
        for (int k = 0; k < (n + 3) / 4; ++k) {
          const uint4 x = reinterpret_cast<const uint4*>(sLength)[k];
          place += (x.x > key) + (x.y > key) + (x.z > key) + (x.w > key);
        }
        sOrder[place] = (uint16_t)t;
      }
    }
  }
  if constexpr (kPackedDirect) {
    constexpr int kWarps = C::kThreads / 32, kRounds = (kMaxWords + kWarps - 1) / kWarps;
    int rk[kRounds];
#pragma unroll
    for (int t = 0; t < kRounds; ++t) {
      const int j = (warp + t * kWarps) * 32 + lane;
      rk[t] = j < p.NB ? p.rank[j] : -1;
    }
#pragma unroll
    for (int t = 0; t < kRounds; ++t) {
      const int w = warp + t * kWarps;
      if (w < p.Wd) {
        sRank[w * 32 + lane] = (uint8_t)((unsigned)rk[t] < (unsigned)p.P ? rk[t] : 0xff);
        for (int r = 0; r < p.P; ++r) {
          const uint32_t word = __ballot_sync(0xffffffffu, rk[t] == r);
          if (lane == 0) sOwn[r * p.Wd + w] = word;
        }
      }
    }
    // More items than CTAs, because the consumer has more than its share of the blocks: every CTA puts them in order by
    // counting their lengths.  An item is a block or two neighbours, a thread has up to kPer.  Items of one length
    // stay in order of their numbers: all CTAs have to come to the same order.
    int n_own = 0, per_head = 0, n = p.BH * ((p.NB + C::kEPT - 1) / C::kEPT);
    if (n > (int)gridDim.x) {  // (as many as if all blocks were the consumer's)
#pragma unroll
      for (int t = 0; t < kRounds; ++t)
        if (t * C::kThreads < p.NB) n_own += __syncthreads_count(rk[t] == p.consumer);
      per_head = (n_own + C::kEPT - 1) / C::kEPT;
      n = p.BH * per_head;
    }
    if (n > (int)gridDim.x) {
      const uint32_t own = lane < p.Wd ? sOwn[p.consumer * p.Wd + lane] : 0u;
      const int own_before = bits_below(own, lane, &n_own);
      // [NB + 1] place NB - length: items of that length, then where they begin
      int* at = reinterpret_cast<int*>(smem + C::kOffEnt);
      uint16_t* blocks = reinterpret_cast<uint16_t*>(smem + C::kOffFirst);
      for (int t = tid; t <= p.NB; t += C::kThreads) at[t] = 0;
      for (int w = warp; w < p.Wd; w += kWarps) {  // (the same for all lanes)
        const uint32_t word = __shfl_sync(0xffffffffu, own, w);
        const int first = __shfl_sync(0xffffffffu, own_before, w);
        if ((word >> lane) & 1u) blocks[first + __popc(word & ((1u << lane) - 1u))] = (uint16_t)(w * 32 + lane);
      }
      __syncthreads();
      constexpr int kPer = (kMaxPackedDirect + C::kThreads - 1) / C::kThreads;
      int place[kPer];  // NB - length, -1 where there is no item
      uint32_t peers[kPer];
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int t = tid + u * C::kThreads;
        place[u] = -1;
        if (t < n) {
          const int bh = t / per_head, x = (t - bh * per_head) * C::kEPT;
          const uint32_t* rows = p.mask + (int64_t)bh * p.NB * p.Wd;
          const uint32_t* row0 = rows + blocks[x] * p.Wd;
          const uint32_t* row1 = rows + blocks[min(x + C::kEPT - 1, n_own - 1)] * p.Wd;
          int left = p.NB;
#pragma unroll 8
          for (int w = 0; w < p.Wd; ++w) left -= __popc(C::kStacked ? row0[w] | row1[w] : row0[w]);
          place[u] = max(left, 0);  // (a mask has no bits behind its NB-th)
        }
        peers[u] = __match_any_sync(0xffffffffu, place[u]);
        if (t < n && lane == __ffs(peers[u]) - 1) atomicAdd(at + place[u], __popc(peers[u]));
      }
      __syncthreads();
      if (warp == 0) {
        int before = 0;
        for (int t0 = 0; t0 <= p.NB; t0 += 32) {  // (the same for all lanes)
          const int count = t0 + lane <= p.NB ? at[t0 + lane] : 0;
          int incl = count;
#pragma unroll
          for (int s = 1; s < 32; s <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, s);
            if (lane >= s) incl += v;
          }
          if (t0 + lane <= p.NB) at[t0 + lane] = before + incl - count;
          before += __shfl_sync(0xffffffffu, incl, 31);
        }
      }
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        const int t = tid + u * C::kThreads, leader = __ffs(peers[u]) - 1;
        for (int k = 0; k < kWarps && u * C::kThreads + k * 32 < n; ++k) {  // warp by warp
          __syncthreads();
          if (warp == k) {
            int first = 0;
            if (t < n && lane == leader) {
              first = at[place[u]];
              at[place[u]] = first + __popc(peers[u]);
            }
            first = __shfl_sync(0xffffffffu, first, leader);
            if (t < n) sOrder[first + __popc(peers[u] & ((1u << lane) - 1u))] = (uint16_t)t;
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;

  // the utility warpgroups hand most of their registers to the softmax warpgroups (the re-balancing
  // instruction sits inside each role's branch so that the register allocator sees which code runs
  // under which limit)
  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SPARSP_REGS_UTILITY));
    // K (of_v = 0) or V tile n of an item's list; an absent second half re-reads the last entry
    auto load_kv = [&](const CUtensorMap* tm, uint64_t* bar, unsigned char* dst, const EntT* ent, int n, int n_ent,
                       int head, int batch, int of_v) {
#pragma unroll
      for (int e = 0; e < C::kEPT; ++e) {
        const uint32_t v = ent[min(n * C::kEPT + e, n_ent - 1)];
        bool remote = false;
        if constexpr (kPacked) {
          remote = (v & E::kRemote) != 0u;
          if (remote) {
            // a remote block's K tile and V tile are consecutive tiles of the consumer's packed buffer
#pragma unroll
            for (int c = 0; c < D / 64; ++c)
              tma_load_4d(dst + c * 16384 + e * (BLK * 128), &tmP, bar, c * 64, 0, (int)(v & E::kValue) + of_v, 0);
          }
        }
        if (!remote) {
          const int tok = (int)(v & (kMaxBlocks - 1)) * BLK;
#pragma unroll
          for (int c = 0; c < D / 64; ++c)
            tma_load_4d(dst + c * 16384 + e * (BLK * 128), tm, bar, c * 64, tok, head, batch);
        }
      }
    };
    if (warp == 3) {
      // ================================ TMA producer: V =====================================
      if (lane == 0) {
        int vn = 0;  // V tiles loaded so far
        for (int i = 0;; ++i) {
          const int buf = i % kLists;
          mbar_wait_bounded_inline(list_ready + buf, (i / kLists) & 1, s_abort, 58, p.wait_limit);
          const int4 hd = s_head[buf];
          if (hd.y == 0) break;  // (only the list builder decides when to stop: all roles stop at the same item)
          const int n_ent = hd.y & kHeadEntries, n_tiles = (n_ent + C::kEPT - 1) / C::kEPT;
          const int batch = hd.w, head = hd.x - batch * p.H;
          const EntT* ent = sEnt + buf * kMaxBlocks;
          for (int n = 0; n < n_tiles; ++n, ++vn) {
            const int st = vn % SV;
            mbar_wait_bounded_inline(v_empty + st, ((vn / SV) & 1) ^ 1, s_abort, 59, p.wait_limit);
            mbar_expect_tx(v_full + st, C::kTileBytes);
            load_kv(&tmV, v_full + st, sV + st * C::kTileBytes, ent, n, n_ent, head, batch, 1);
          }
          mbar_arrive(list_free + buf);
        }
      }
    } else if (warp == 0) {
      // ================================ TMA producer: Q and K ===============================
      if (lane == 0) {
        QKRing<C::kStagesK> at;
        for (int i = 0;; ++i) {
          const int buf = i % kLists;
          mbar_wait_bounded_inline(list_ready + buf, (i / kLists) & 1, s_abort, 51, p.wait_limit);
          const int4 hd = s_head[buf];
          if (hd.y == 0) break;  // (only the list builder decides when to stop: all roles stop at the same item)
          const int n_ent = hd.y & kHeadEntries, n_tiles = (n_ent + C::kEPT - 1) / C::kEPT;
          const int batch = hd.w, head = hd.x - batch * p.H;
          const EntT* ent = sEnt + buf * kMaxBlocks;
          {
            // a Q tile is 128 rows: one 128-token block, or two 64-token blocks stacked (an absent second
            // block re-reads the first: finite data whose rows are never used)
            const uint32_t b = at.next_q();
            mbar_wait_bounded_inline(qk_empty + b, at.use(b) ^ 1u, s_abort, 52, p.wait_limit);
            mbar_expect_tx(qk_full + b, C::kTileBytes);
#pragma unroll
            for (int q = 0; q < C::kEPT; ++q) {
              const int b1 = (int)((uint32_t)hd.z >> 16), bq = q && b1 != 0xffff ? b1 : hd.z & 0xffff;
#pragma unroll
              for (int c = 0; c < D / 64; ++c)
                tma_load_4d(sQK + b * C::kTileBytes + c * 16384 + q * (BLK * 128), &tmQ, qk_full + b, c * 64, bq * BLK,
                            head, batch);
            }
          }
          for (int n = 0; n < n_tiles; ++n) {
            const uint32_t b = at.next_k();
            mbar_wait_bounded_inline(qk_empty + b, at.use(b) ^ 1u, s_abort, 57, p.wait_limit);
            mbar_expect_tx(qk_full + b, C::kTileBytes);
            load_kv(&tmK, qk_full + b, sQK + b * C::kTileBytes, ent, n, n_ent, head, batch, 0);
          }
          mbar_arrive(list_free + buf);
        }
      }
    } else if (warp == 1) {
      // ================================ Q K^T issuer ========================================
      // The whole warp runs the loop (uniform control flow and operands); one elected lane issues.
      const bool leader = elect_one();
      constexpr uint32_t kIdescQK = make_idesc_bf16(128, 128, 0, 0);
      const uint64_t desc0 = make_smem_desc(smem_u32(sQK), 16, 1024);
      const uint32_t hi = (uint32_t)(desc0 >> 32);
      uint32_t lo[D / 16];
#pragma unroll
      for (int kk = 0; kk < D / 16; ++kk)
        lo[kk] = (uint32_t)desc0 + (uint32_t)(((kk / 4) * 16384 + (kk % 4) * 32) >> 4);
      QKRing<C::kStagesK> at;
      int g = 0, w = 0;     // tiles so far, the next one's warpgroup
      uint32_t round = 0u;  // parity of that warpgroup's tiles so far
      for (int i = 0;; ++i) {
        const int buf = i % kLists;
        mbar_wait_bounded_inline(list_ready + buf, (i / kLists) & 1, s_abort, 53, p.wait_limit);
        const int y = s_head[buf].y;
        if (y == 0) break;
        const int n_tiles = ((y & kHeadEntries) + C::kEPT - 1) / C::kEPT;
        const uint32_t bq = at.next_q();
        mbar_wait_bounded_inline(qk_full + bq, at.use(bq), s_abort, 11, p.wait_limit);
        const uint32_t q_off = bq * (C::kTileBytes >> 4);
        for (int n = 0; n < n_tiles; ++n, ++g) {
          const uint32_t bk = at.next_k();
          mbar_wait_bounded_inline(qk_full + bk, at.use(bk), s_abort, 12, p.wait_limit);
          // an S buffer is free once its warpgroup has loaded the scores of its tile before, or the P V has read the P
          // that took their place
          if (g >= C::kWGs) {
            if (C::kInPlaceP)
              mbar_wait_bounded_inline(o_full + ((g - C::kWGs) & 3), ((g - C::kWGs) >> 2) & 1, s_abort, 24,
                                       p.wait_limit);
            else
              mbar_wait_bounded_inline(s_free + w, round ^ 1u, s_abort, 24, p.wait_limit);
          }
          tc_fence_after();
          const uint32_t k_off = bk * (C::kTileBytes >> 4);
          const uint32_t tS = tmem_base + C::kColS + w * 128;
          if (leader) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              mma_ss_lohi(tS, lo[kk] + q_off, hi, lo[kk] + k_off, hi, kIdescQK, kk > 0 ? 1u : 0u);
            mma_commit(s_full + w);
            mma_commit(qk_empty + bk);
            if (n == n_tiles - 1) mma_commit(qk_empty + bq);
          }
          __syncwarp();
          if (++w == C::kWGs) {
            w = 0;
            round ^= 1u;
          }
        }
        if (lane == 0) mbar_arrive(list_free + buf);
        __syncwarp();
      }
    } else {
      // ================================ P V issuer ==========================================
      const bool leader = elect_one();
      constexpr uint32_t kIdescPV = make_idesc_bf16(128, C::kAccCols, 0, 1);
      // second 64-column group of the B operand: the other half of a d = 128 tile, or the block of ones, which
      // lies kOffOnes - kOffV behind the FIRST stage (the stage offset is taken off again below)
      const uint64_t descV = make_smem_desc(smem_u32(sV), C::kOnes ? (uint32_t)(C::kOffOnes - C::kOffV) : 16384u, 1024);
      const uint32_t hiV = (uint32_t)(descV >> 32);
      uint32_t vlo[8];
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) vlo[kk] = (uint32_t)descV + (uint32_t)((kk * 2048) >> 4);
      const uint32_t tO = tmem_base + C::kColO;
      constexpr uint32_t kIdescSum = make_idesc_bf16(128, 16, 0, 1);
      const uint64_t descOnes = make_smem_desc(smem_u32(smem + C::kOffOnes), 16384u, 1024);
      const uint32_t tL = tmem_base + C::kColL;
      int g = 0, w = 0;
      uint32_t round = 0u;
      for (int i = 0;; ++i) {
        const int buf = i % kLists;
        mbar_wait_bounded_inline(list_ready + buf, (i / kLists) & 1, s_abort, 54, p.wait_limit);
        const int y = s_head[buf].y;
        if (y == 0) break;
        const int n_tiles = ((y & kHeadEntries) + C::kEPT - 1) / C::kEPT;
        // the previous item's accumulator must have been read out before this item's first P V overwrites it
        if (i > 0) mbar_wait_bounded_inline(o_drained, (i - 1) & 1, s_abort, 55, p.wait_limit);
        for (int n = 0; n < n_tiles; ++n, ++g) {
          mbar_wait_bounded_inline(p_full + w, round, s_abort, 20, p.wait_limit);
          mbar_wait_bounded_inline(v_full + g % SV, (g / SV) & 1, s_abort, 22, p.wait_limit);
          tc_fence_after();
          uint32_t stage_off = (uint32_t)(((g % SV) * C::kTileBytes) >> 4);
          if (C::kOnes) stage_off -= stage_off << 16;  // start address up, distance to the ones block down
          const uint32_t tP = tmem_base + (C::kInPlaceP ? C::kColS + w * 128 : C::kColP);
          if (leader) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
              mma_ts_lohi(tO, tP + kk * 8, vlo[kk] + stage_off, hiV, kIdescPV, (kk > 0 || n > 0) ? 1u : 0u);
              if (C::kSum128)
                mma_ts_lohi(tL, tP + kk * 8, (uint32_t)descOnes, (uint32_t)(descOnes >> 32), kIdescSum,
                            (kk > 0 || n > 0) ? 1u : 0u);
            }
            mma_commit(o_full + (g & 3));
            mma_commit(v_empty + g % SV);
          }
          __syncwarp();
          if (++w == C::kWGs) {
            w = 0;
            round ^= 1u;
          }
        }
        if (lane == 0) mbar_arrive(list_free + buf);
        __syncwarp();
      }
    }
  } else if (warp < 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(SPARSP_REGS_UTILITY2));
    // ================================ list builder ========================================
    if (warp == 4) {
      // union of the item's (up to) two mask rows -> ascending entry list; flag bit q = kept by query
      // block blk[q].  Runs up to two items ahead of the consumers.
      // Items are handed out head by head (a head's K and V stay in L2).  A CTA's first item is its own number, the
      // following ones come from a global counter (first come, first served), so CTAs whose items are short simply take
      // more of them; the head travels to the other roles with the list.
      // Packed source: a head has few items, the consumer's; they are numbered without gaps, and since numbers only
      // grow the place of an item is found by walking the heads' item counts forward, 32 heads at a time with a count
      // per lane. K / V source: all query blocks count, and nearly always all of them keep something.
      int hb = 0, hbase = 0, h_end;  // first head of the 32, items before it, items up to and including this lane's
      auto load_heads = [&]() {
        h_end = hb + lane < p.BH ? p.n_items[hb + lane] : 0;
#pragma unroll
        for (int s = 1; s < 32; s <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, h_end, s);
          if (lane >= s) h_end += v;
        }
        h_end += hbase;
      };
      if (kSource == Source::kPacked) load_heads();
      // kPackedDirect: the consumer's blocks, a word per lane, and how many of them lie in lower words
      uint32_t own = 0u;
      int n_own = 0, own_before = 0, number = 0, first_of = -1, base_of = -1, own_base = 0;
      if constexpr (kPackedDirect) {
        own = lane < p.Wd ? sOwn[p.consumer * p.Wd + lane] : 0u;
        own_before = bits_below(own, lane, &n_own);
      }
      auto own_block = [&](int x) {  // the consumer's x-th block
        const int w = 31 - __clz(__ballot_sync(0xffffffffu, own != 0u && own_before <= x));
        uint32_t left = __shfl_sync(0xffffffffu, own, w);
        for (int skip = x - __shfl_sync(0xffffffffu, own_before, w); skip > 0; --skip) left &= left - 1u;
        return w * 32 + __ffs(left) - 1;
      };
      int bh = p.BH, blk0 = -1, blk1 = -1;
      const int ragged_block = p.N % BLK ? p.NB - 1 : -1;
      uint32_t rb0 = 0u, rb1 = 0u;  // the item's mask rows, a word per lane (NB <= 1024: at most 32 words)
      // Takes an item: its head (BH = no more items), query block(s) and mask rows.
      auto load_rows = [&]() {
        const uint32_t* rows = p.mask + (int64_t)bh * p.NB * p.Wd;
        rb0 = lane < p.Wd ? rows[blk0 * p.Wd + lane] : 0u;
        rb1 = lane < p.Wd && blk1 >= 0 ? rows[blk1 * p.Wd + lane] : 0u;
      };
      auto fetch = [&](int it) {
        if constexpr (kDirect || kPackedDirect) {  // the CTAs take places from the front and from behind in turn
          const int per_head = kDirect ? p.NB : (n_own + C::kEPT - 1) / C::kEPT, n = p.BH * per_head;
          bh = p.BH;
          if (it >= n) return;
          const int item = n > (int)gridDim.x ? sOrder[it] : it, at = item / per_head, x = item - at * per_head;
          bh = at;
          blk0 = kDirect ? x : own_block(x * C::kEPT);
          blk1 = kPackedDirect && C::kStacked && x * C::kEPT + 1 < n_own ? own_block(x * C::kEPT + 1) : -1;
          load_rows();
          if (!__any_sync(0xffffffffu, (rb0 | rb1) != 0u)) bh = p.BH;  // (and so do all behind it)
          return;
        }
        int x;
        if (kPacked) {
          uint32_t after;  // heads whose items end behind this one
          while ((after = __ballot_sync(0xffffffffu, it < h_end)) == 0u && hb + 32 < p.BH) {
            hbase = __shfl_sync(0xffffffffu, h_end, 31);
            hb += 32;
            load_heads();
          }
          const int f = __ffs(after) - 1;
          bh = after ? hb + f : p.BH;
          x = it - (f > 0 ? __shfl_sync(0xffffffffu, h_end, f - 1) : hbase);
        } else {
          // Behind a head's last item are its query blocks that keep nothing: all CTAs go on with the next head.
          auto leave_head = [&](int first) {
            int to = 0;
            if (lane == 0) {
              atomicMax(p.work_counter, max(first - (int)gridDim.x, 0));
              to = (int)gridDim.x + atomicAdd(p.work_counter, 1);
            }
            return __shfl_sync(0xffffffffu, to, 0);
          };
          bh = find_item(it, C::kStacked ? (p.NB + 1) / 2 : p.NB, p.BH, p.n_items, leave_head,
                         [&] { return *s_abort != 0; }, &x);
        }
        if (bh >= p.BH) return;
        const int32_t* items = p.pairs + (int64_t)bh * (2 * ((p.NB + 1) / 2));
        blk0 = C::kStacked ? items[2 * x] : items[x];
        blk1 = C::kStacked ? items[2 * x + 1] : -1;
        load_rows();
      };
      auto next_item = [&]() {
        if (kDirect || kPackedDirect) {
          const int turn_no = ++number, c = (int)blockIdx.x, G = (int)gridDim.x;
          return turn_no * G + (turn_no & 1 ? G - 1 - c : c);
        }
        int it = 0;
        if (lane == 0) it = (int)gridDim.x + atomicAdd(p.work_counter, 1);
        return __shfl_sync(0xffffffffu, it, 0);
      };
      // An item that has failed is handed out again.  Its verdict is there once its list buffer is free: before the
      // buffer is used again, or, when there are no more items, one outstanding item after the other.
      int checked = 0;  // items whose verdict has been seen
      int meetings = 0;  // items so far whose rows are written behind a meeting
      auto verdict = [&]() -> int {
        const int b = checked % kLists;
        mbar_wait_bounded_inline(list_free + b, (checked / kLists) & 1, s_abort, 50, p.wait_limit);
        ++checked;
        return s_failed[b] ? b : -1;
      };
      for (int i = 0;; ++i) {
        const int buf = i % kLists;
        int again = -1;  // list buffer of an item that is computed again now (rare)
        if (checked <= i - kLists) again = verdict();
        if (again < 0) fetch(i == 0 ? (int)blockIdx.x : next_item());
        while (again < 0 && bh >= p.BH && checked < i) again = verdict();
        if (__any_sync(0xffffffffu, *s_abort != 0) || (again < 0 && bh >= p.BH)) {
          if (lane == 0) {
            s_head[buf].y = 0;
            mbar_arrive(list_ready + buf);
          }
          break;
        }
        const int next_bh = bh;
        if (again >= 0) {
          bh = s_head[again].x;
          const int z = s_head[again].z;
          blk0 = z & 0xffff;
          blk1 = (int)((uint32_t)z >> 16) == 0xffff ? -1 : (int)((uint32_t)z >> 16);
          load_rows();
          __syncwarp();  // (every lane has looked)
          if (lane == 0) s_failed[again] = 0;
        }
        EntT* ent = sEnt + buf * kMaxBlocks;
        const int batch = bh / p.H;
        if constexpr (kPackedDirect) {
          if (batch != base_of) {  // the consumer's first tile
            const int64_t br = (int64_t)batch * p.P + p.consumer;
            int64_t first = 0;
            if (p.dst_base) {
              first = p.dst_base[br] / p.tile_bytes;
            } else {
              for (int64_t t = lane; t < br; t += 32) first += 2 * p.seg_total[t];
#pragma unroll
              for (int s = 16; s >= 1; s >>= 1) first += __shfl_xor_sync(0xffffffffu, first, s);
            }
            own_base = (int)first;
            base_of = batch;
          }
          if (bh != first_of) {  // places of the head's blocks: of every producer, the entries before each word's
            const int64_t br = (int64_t)batch * p.P + p.consumer, h = bh - batch * p.H;
            const uint32_t u = lane < p.Wd ? p.U[(br * p.H + h) * p.Wd + lane] : 0u;
            const int64_t* off = p.seg_off + br * p.P * p.H + h;
            const int o0 = lane < p.P ? (int)off[(int64_t)lane * p.H] : 0;
            const int o1 = lane + 32 < p.P ? (int)off[(int64_t)(lane + 32) * p.H] : 0;
            int32_t* first = reinterpret_cast<int32_t*>(smem + C::kOffFirst);
            for (int r = 0; r < p.P; ++r) {
              int total;
              const int below = bits_below(lane < p.Wd ? u & sOwn[r * p.Wd + lane] : 0u, lane, &total);
              const int o = __shfl_sync(0xffffffffu, r < 32 ? o0 : o1, r & 31);
              if (lane < p.Wd) first[r * p.Wd + lane] = o + below;
            }
            if (lane < p.Wd) reinterpret_cast<uint32_t*>(smem + C::kOffUnion)[lane] = u;
            __syncwarp();
            first_of = bh;
          }
        }
        const int tile_base = kPackedDirect ? own_base : kPacked ? (int)p.tile_base[batch] : 0;
        // Entry order (any order gives the same attention).  Blocks BOTH query blocks keep make full tiles; a
        // block only the first keeps is put next to a block only the second keeps, so that such a tile costs
        // every softmax row one 64-key half instead of costing half of the rows two.  A full tile is bound by
        // the softmax warps, a half-work tile by the tensor pipe (its MMAs cost the same), so the two kinds
        // alternate in groups of two tiles (one of each per softmax warpgroup) while both last; then the rest
        // of the full tiles, the rest of the paired one-sided blocks and what is left of the longer one-sided
        // list.  With a single query block this is plain ascending order.
        // A mask word at a time, a lane per bit: next to busy softmax warps an instruction of this warp gets issued
        // every several cycles, so the list is as late as it has instructions.
        const uint32_t below = (1u << lane) - 1u;
        // Packed source: the item's own query blocks come first.  There a row meets the largest score that it is likely
        // to meet, so the reference it takes from the first tile makes that term's exponential exactly 1 (24 heads x
        // 24576, 4 ranks: 1.87e-3 from 64 bits; 2.00e-3 with the first tile as it comes, 1.95e-3 with a reference that
        // follows the maximum).
        int lead = 0, own_of = 0;  // entries ahead of the classes; bit q: one of them is kept by query block q
        int rag_pos = -1;          // where the sequence's ragged last block went
        if (kPacked) {
#pragma unroll
          for (int q = 0; q < (C::kStacked ? 2 : 1); ++q) {
            const int j = q ? blk1 : blk0;
            if (j < 0) continue;
            const uint32_t f0 = __shfl_sync(0xffffffffu, rb0, j >> 5), f1 = __shfl_sync(0xffffffffu, rb1, j >> 5);
            const uint32_t f = ((f0 >> (j & 31)) & 1u) | ((f1 >> (j & 31)) & 1u) << 1;
            if (f == 0u) continue;
            if (lane == (j >> 5)) {
              rb0 &= ~(1u << (j & 31));
              rb1 &= ~(1u << (j & 31));
            }
            own_of |= (int)f;
            if (lane == 0) ent[lead] = (EntT)((uint32_t)j | f << E::kFlagShift);
            if (j == ragged_block) rag_pos = lead;
            ++lead;
          }
        }
        int n_both = 0, n_mix = 0, n_grp = 0, running, none = 0;
        if (C::kStacked) {
          n_both = __reduce_add_sync(0xffffffffu, __popc(rb0 & rb1));
          const int n0 = __reduce_add_sync(0xffffffffu, __popc(rb0 & ~rb1));
          const int n1 = __reduce_add_sync(0xffffffffu, __popc(rb1 & ~rb0));
          n_mix = min(n0, n1);
          // two full tiles (four blocks both keep), then two half-work tiles (two one-sided pairs), and so on
          n_grp = min(n_both >> 2, n_mix >> 1);
          running = lead + n_both + n0 + n1;
          none = (n_both + n0 == 0 ? 1 : 0) | (n_both + n1 == 0 ? 2 : 0);
          none &= ~own_of;
        } else {
          running = lead + __reduce_add_sync(0xffffffffu, __popc(rb0));
        }
        int at0 = 0, at1 = 0, at2 = 0;  // entries of each class so far
        for (uint32_t todo = __ballot_sync(0xffffffffu, (rb0 | rb1) != 0u); todo; todo &= todo - 1) {
          const int w = __ffs(todo) - 1;
          const uint32_t w0 = __shfl_sync(0xffffffffu, rb0, w);
          const uint32_t w1 = C::kStacked ? __shfl_sync(0xffffffffu, rb1, w) : 0u;
          const int jb = w * 32 + lane;
          if (C::kStacked) {
            const uint32_t both = w0 & w1, only0 = w0 & ~w1, only1 = w1 & ~w0;
            const bool in0 = (w0 >> lane) & 1u, in1 = (w1 >> lane) & 1u;
            if (in0 || in1) {
              int pos;
              if (in0 && in1) {
                const int idx = at0 + __popc(both & below);
                pos = idx < 4 * n_grp ? 8 * (idx >> 2) + (idx & 3) : 4 * n_grp + idx;
              } else {
                const int c = in0 ? 0 : 1, idx = in0 ? at1 + __popc(only0 & below) : at2 + __popc(only1 & below);
                if (idx < 2 * n_grp) pos = 8 * (idx >> 1) + 4 + 2 * (idx & 1) + c;
                else if (idx < n_mix) pos = n_both + 2 * idx + c;
                else pos = n_both + n_mix + idx;  // tail of the longer class
              }
              pos += lead;
              ent[pos] = (EntT)((uint32_t)jb | ((in0 ? 1u : 0u) | (in1 ? 2u : 0u)) << E::kFlagShift);
              if (jb == ragged_block) rag_pos = pos;
            }
            at0 += __popc(both);
            at1 += __popc(only0);
            at2 += __popc(only1);
          } else {
            if ((w0 >> lane) & 1u) {
              const int pos = lead + at0 + __popc(w0 & below);
              ent[pos] = (EntT)((uint32_t)jb | 1u << E::kFlagShift);
              if (jb == ragged_block) rag_pos = pos;
            }
            at0 += __popc(w0);
          }
        }
        __syncwarp();
        // the softmax code lets only the LAST tile reach past the end of the sequence: if the last block of
        // the sequence is ragged and in the list, it trades places with the last entry
        rag_pos = __reduce_max_sync(0xffffffffu, rag_pos);
        if (rag_pos >= 0) {
          if (lane == 0) {
            const int e = running - 1;
            const EntT t = ent[rag_pos];
            ent[rag_pos] = ent[e];
            ent[e] = t;
          }
          __syncwarp();
        }
        if (C::kStacked && (running & 1) && lane == 0) ent[running] = 0;
        if constexpr (kPacked) {  // where the entries' blocks are, a lane per entry, two loads in flight
          const int32_t* slot = p.slot + (int64_t)bh * p.NB;
          auto slot_of = [&](int j) -> int32_t {
            if constexpr (kPackedDirect) {
              const int r = sRank[j], w = j >> 5;
              if (r >= p.P || r == p.consumer) return -1;
              const uint32_t set = reinterpret_cast<const uint32_t*>(smem + C::kOffUnion)[w] & sOwn[r * p.Wd + w];
              if (!((set >> (j & 31)) & 1u)) return -1;
              const int32_t* first = reinterpret_cast<const int32_t*>(smem + C::kOffFirst);
              return first[r * p.Wd + w] + __popc(set & ((1u << (j & 31)) - 1u));
            } else {
              return slot[j];
            }
          };
          auto placed_at = [&](uint32_t v, int32_t sl) {
            return sl < 0 ? v : (v & ~E::kValue) | E::kRemote | ((uint32_t)(tile_base + 2 * sl) & E::kValue);
          };
          for (int e = lane; e < running; e += 64) {
            const bool two = e + 32 < running;
            const uint32_t v1 = ent[e], v2 = two ? ent[e + 32] : v1;
            const int32_t s1 = slot_of(v1 & (kMaxBlocks - 1)), s2 = slot_of(v2 & (kMaxBlocks - 1));
            ent[e] = placed_at(v1, s1);
            if (two) ent[e + 32] = placed_at(v2, s2);
          }
          __syncwarp();
        }
        int ref_of = kPacked || running <= (kZeroMinTiles - 1) * C::kEPT ? kRefFirst : kRefZero;
        if (again >= 0) ref_of = kRefExact;
        int meet = 0;
        if (p.in_place || again >= 0) meet = kHeadMeet | (meetings++ & 1) << kHeadMeetParityShift;
        if (lane == 0) {
          s_head[buf] = make_int4(bh, running | (rag_pos >= 0 ? kHeadRagged : 0) | ref_of << kHeadRefShift |
                                          none << kHeadNoneShift | meet,
                                  blk0 | (blk1 < 0 ? 0xffff : blk1) << 16, batch);
          s_failed[buf] = 0;
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(list_ready + buf);
        if (again >= 0) bh = next_bh;  // (>= BH where there are no more items)
      }
    } else {
      // ============== rows of query blocks that keep nothing, which are no work items ==============
      // They have nothing to do with the items, so three idle warps write them while the others work: 677 MB of an
      // attention of 40 heads x 75600 to one rank's own blocks.  A lane looks at a query block of its own, since a look
      // is one or two loads that wait for each other; neighbours go to different warps.
      // (They are alone with it where hardly anything is kept, so no 64-bit division is in their way: nothing kept by
      // 16 heads x 591 blocks of 128 x 64 is 49.5 us a call; 76.9 with such divisions, 16-byte stores and a sort of no
      // items.)
      const unsigned n_rows = (unsigned)p.BH * p.NB, warps = gridDim.x * 3, mine = blockIdx.x * 3 + warp - 5;
      for (unsigned u0 = mine; u0 < n_rows; u0 += 32 * warps) {
        const unsigned u = u0 + lane * warps;  // (batch, head, block)
        bool empty = u < n_rows && (!kPacked || p.rank[u % (unsigned)p.NB] == p.consumer);
        if (empty) {
          const uint32_t* row = p.mask + (int64_t)u * p.Wd;
          uint32_t any = 0;
#pragma unroll 8
          for (int w = 0; w < p.Wd; ++w) any |= row[w];
          empty = any == 0u;
        }
        for (uint32_t todo = __ballot_sync(0xffffffffu, empty); todo; todo &= todo - 1) {
          const unsigned v = u0 + (__ffs(todo) - 1) * warps, bh = v / (unsigned)p.NB;
          clear_rows<D, BLK>(p, (int)bh, (int)(v - bh * p.NB));
        }
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(C::kRegsSoftmax));
    // ================================ softmax warpgroups ==================================
    const int wg = (warp >> 2) - 2;  // takes the tiles with g % kWGs = wg, in S buffer wg
    const int rgrp = warp & 3;       // tensor-memory lane group this warp may access
    const int row = rgrp * 32 + lane;
    const int rh = row >> 6;         // which query block of a stacked Q tile the row belongs to
    const uint32_t lane_off = (uint32_t)(rgrp * 32) << 16;
    const uint32_t tS = tmem_base + C::kColS + wg * 128 + lane_off;
    const uint32_t tP = C::kInPlaceP ? tS : tmem_base + C::kColP + lane_off;
    const uint32_t tO = tmem_base + C::kColO + lane_off;
    // the warps of a row group: mine, and the one that takes the tiles before mine
    const int mine = wg * 4 + rgrp, before = (wg == 0 ? C::kWGs - 1 : wg - 1) * 4 + rgrp;
    int g0 = 0, w0 = 0;     // number of the item's first tile, its warpgroup
    uint32_t round = 0u;    // parity of my tiles so far
    int turns = 0, given = 0;  // turns taken over from the warp before and handed to the one behind so far
    for (int i = 0;; ++i) {
      const int buf = i % kLists;
      mbar_wait_bounded_inline(list_ready + buf, (i / kLists) & 1, s_abort, 56, p.wait_limit);
      const int4 hd = s_head[buf];
      if (hd.y == 0) break;
      const int n_ent = hd.y & kHeadEntries;
      const int n_tiles = (n_ent + C::kEPT - 1) / C::kEPT;
      const int first = wg >= w0 ? wg - w0 : wg - w0 + C::kWGs;  // my first tile
      const int ref_of = (hd.y >> kHeadRefShift) & 3;
      const EntT* ent = sEnt + buf * kMaxBlocks;
      const bool item_ragged = (hd.y & kHeadRagged) != 0;
      volatile float* ref = sRef + (i & 3) * 128;
      float m_ref = ref_of == kRefZero ? 0.0f : -INFINITY;  // the row's reference as this thread last saw it
      float i_max = 0.0f;  // largest binary exponent that was taken on the FMA pipe, in magnitude
      bool exact = ref_of == kRefExact;  // this row group takes the running maximum
      auto learn_ref = [&]() {  // the warpgroup that does not own the first tile
        mbar_wait_bounded_inline(ref_ready + (i & 3), (i >> 2) & 1, s_abort, 43, p.wait_limit);
        exact = s_exact[(i & 3) * 4 + rgrp] != 0;
        if (ref_of == kRefFirst && !exact) m_ref = ref[row];
      };
      auto take_turn = [&]() {  // the other warp has decided about the tile before, and may have moved the reference
        mbar_wait_bounded_inline(turn + before + (turns & 1) * 4 * C::kWGs, (turns >> 1) & 1, s_abort, 44,
                                 p.wait_limit);
        ++turns;
        m_ref = ref[row];
      };
      auto give_turn = [&]() { mbar_arrive(turn + mine + (given++ & 1) * 4 * C::kWGs); };
      // the row's largest score of a tile: one flat instruction stream per 64-key half, an absent half (not kept by
      // this row's query block) is skipped
      auto row_max = [&](const float* sv, const int* vh) {
        float mx = -INFINITY;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float* svh = sv + h * 64;
          if (vh[h] > 0) {
            float m0 = svh[0], m1 = svh[1], m2 = svh[2], m3 = svh[3];
#pragma unroll
            for (int e = 4; e < 64; e += 4) {
              m0 = fmaxf(m0, svh[e]);
              m1 = fmaxf(m1, svh[e + 1]);
              m2 = fmaxf(m2, svh[e + 2]);
              m3 = fmaxf(m3, svh[e + 3]);
            }
            mx = fmaxf(mx, fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)));
          }
        }
        return mx * p.scale_log2;
      };
      // the warpgroup that does
      auto look_at_first = [&](auto careful_tag, const float* sv, const int* vh) {
        if ((decltype(careful_tag)::value || kPacked) && ref_of == kRefFirst) {
          const float mx = row_max(sv, vh);
          m_ref = mx > -INFINITY ? mx : 0.0f;  // (keeps nothing of this tile, or is no number)
          ref[row] = m_ref;
          exact = __any_sync(0xffffffffu, !(fabsf(m_ref) <= kFirstSample));
        } else {
          float most = 0.0f;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (vh[h] > 0) {
#pragma unroll
              for (int e = h * 64; e < h * 64 + 64; e += 16) most = max_abs3(sv[e], sv[e + 8], most);
            }
          }
          exact = __any_sync(0xffffffffu, !(most * p.scale_log2 <= kZeroSample));
        }
        if (exact) m_ref = -INFINITY;
        __syncwarp();
        if (lane == 0) {
          s_exact[(i & 3) * 4 + rgrp] = exact ? 1 : 0;
          mbar_arrive(ref_ready + (i & 3));
        }
      };

      // The row's reference follows its running maximum; what has been added up so far shrinks by the factor that is
      // returned.
      auto move_ref = [&](const float mx) -> float {
        const float m_new = fmaxf(m_ref, mx);
        const bool grow = m_new > m_ref + kGrowThreshold || (m_ref == -INFINITY && m_new > -INFINITY);
        float alpha = 1.0f;
        if (__any_sync(0xffffffffu, grow)) {
          alpha = grow ? ex2(m_ref - m_new) : 1.0f;  // m_ref = -inf -> 0
          if (grow) {
            m_ref = m_new;
            ref[row] = m_new;
          }
        }
        return alpha;
      };
      // Rescales the row's accumulator, after the exponentials of the tile, which need the new reference only, and
      // before its P is handed over.  Every P V of the item issued so far must have landed in O; they complete in
      // order, so the one of tile g-1 suffices, and the tile behind, which may have a factor of its own by now, waits
      // for the P V of this one.
      auto rescale = [&](const float alpha, const int n) {
        if (n == 0 || !__any_sync(0xffffffffu, alpha != 1.0f)) return;
        const int g = g0 + n;
        mbar_wait_bounded_inline(o_full + ((g - 1) & 3), ((g - 1) >> 2) & 1, s_abort, 38, p.wait_limit);
        tc_fence_after();
        constexpr int kAtOnce = D == 128 ? 64 : 16;  // columns in flight (d = 64 has half the registers)
#pragma unroll 1
        for (int c = 0; c < D / kAtOnce; ++c) {  // the row's accumulator
          uint32_t o[kAtOnce];
#pragma unroll
          for (int q = 0; q < kAtOnce; q += 16) tmem_ld16(tO + c * kAtOnce + q, o + q);
          tmem_ld_wait(o);
#pragma unroll
          for (int e = 0; e < kAtOnce; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
#pragma unroll
          for (int q = 0; q < kAtOnce; q += 16) tmem_st16(tO + c * kAtOnce + q, o + q);
        }
        uint32_t sum[1];  // the row's sum (nobody reads the columns beside it)
        tmem_ld1(tmem_base + C::kColL + lane_off, sum);
        tmem_ld_wait(sum);
        tmem_st1(tmem_base + C::kColL + lane_off, __float_as_uint(__uint_as_float(sum[0]) * alpha));
      };
      // A tile whose P takes the place of its scores: 32 columns at a time, the next ones on their way from tensor
      // memory.
      auto in_place_tile = [&](auto ragged_tag, auto exact_tag, const int n, const int* vh) {
        constexpr bool kRagged = decltype(ragged_tag)::value, kExact = decltype(exact_tag)::value;
        float va[32], vb[32];
        auto load = [&](float(&v)[32], const int q) { tmem_ld32(tS + q * 32, reinterpret_cast<uint32_t*>(v)); };
        auto cut = [&](float(&v)[32], const int q) {  // columns past the end of the sequence count as -inf
          if (kRagged && vh[q >> 1] < 64) {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = (q & 1) * 32 + e < vh[q >> 1] ? v[e] : -INFINITY;
          }
        };
        float alpha = 1.0f;
        if (kExact || n == 0) {  // a look at the whole tile first
          float mx = -INFINITY, most = 0.0f;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (vh[q >> 1] > 0) {
              load(va, q);
              tmem_ld_wait(va);
              cut(va, q);
              if (kExact || ((kRagged || kPacked) && ref_of == kRefFirst)) {
                float m0 = va[0], m1 = va[1];
#pragma unroll
                for (int e = 2; e < 32; e += 2) {
                  m0 = fmaxf(m0, va[e]);
                  m1 = fmaxf(m1, va[e + 1]);
                }
                mx = fmaxf(mx, fmaxf(m0, m1));
              } else {
#pragma unroll
                for (int e = 0; e < 32; e += 16) most = max_abs3(va[e], va[e + 8], most);
              }
            }
          }
          mx *= p.scale_log2;
          if (kExact) {
            if (n > 0) take_turn();
            alpha = move_ref(mx);
            if (n == 0 && m_ref == -INFINITY) ref[row] = m_ref;
            if (n + 1 < n_tiles) give_turn();
          } else {
            if ((kRagged || kPacked) && ref_of == kRefFirst) {
              m_ref = mx > -INFINITY ? mx : 0.0f;  // (keeps nothing of this tile, or is no number)
              ref[row] = m_ref;
              exact = __any_sync(0xffffffffu, !(fabsf(m_ref) <= kFirstSample));
            } else {
              exact = __any_sync(0xffffffffu, !(most * p.scale_log2 <= kZeroSample));
            }
            if (exact) m_ref = -INFINITY;
            __syncwarp();
            if (lane == 0) {
              s_exact[(i & 3) * 4 + rgrp] = exact ? 1 : 0;
              mbar_arrive(ref_ready + (i & 3));
            }
          }
        } else if (n < C::kWGs) {
          learn_ref();
        }
        if (!kExact && n < C::kWGs && exact) return;  // the variant with the turns takes the tile
        const float2 sc2 = make_float2(p.scale_log2, p.scale_log2), nm2 = make_float2(-m_ref, -m_ref);
        auto exponentials = [&](float(&v)[32], const int q) {
          uint32_t pk[16];
          cut(v, q);
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float2 x = ffma2(make_float2(v[2 * e], v[2 * e + 1]), sc2, nm2);
            constexpr int kPoly = SPARSP_TUNE_POLY;
            const float2 pp = (kPoly > 0 && (((q & 1) * 16 + e) % (kPoly > 0 ? kPoly : 1)) == 1)
                                  ? exp2_poly2<kRagged || kExact, !kExact>(x, &i_max)
                                  : make_float2(ex2(x.x), ex2(x.y));
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(pp.x, pp.y);
            pk[e] = *reinterpret_cast<const uint32_t*>(&h2);
          }
          if (kRagged && vh[q >> 1] < 64) {
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              const int c = (q & 1) * 32 + 2 * e;
              pk[e] = c + 1 < vh[q >> 1] ? pk[e] : (c < vh[q >> 1] ? (pk[e] & 0xffffu) : 0u);
            }
          }
          tmem_st16(tP + q * 16, pk);
        };
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (vh[h] > 0) {
            load(va, 2 * h);
            tmem_ld_wait(va);
            load(vb, 2 * h + 1);
            exponentials(va, 2 * h);
            tmem_ld_wait(vb);
            exponentials(vb, 2 * h + 1);
          } else {
            uint32_t none[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) none[e] = 0u;
            tmem_st16(tP + 2 * h * 16, none);
            tmem_st16(tP + (2 * h + 1) * 16, none);
          }
        }
        if (kExact) rescale(alpha, n);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full + wg);
        round ^= 1u;
      };

      // A tile whose P goes to a buffer of its own: the whole row of scores in registers, the S buffer is free at once.
      auto own_buffer_tile = [&](auto ragged_tag, auto exact_tag, const int n, const int* vh) {
        constexpr bool kRagged = decltype(ragged_tag)::value, kExact = decltype(exact_tag)::value;
        const int g = g0 + n;
        float sv[128];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(tS + c * 32, reinterpret_cast<uint32_t*>(sv) + c * 32);
        tmem_ld_wait(sv);
        if (kRagged) {
          // the sequence ends inside this tile: columns past the end count as -inf
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (vh[h] > 0 && vh[h] < 64) {
#pragma unroll
              for (int e = 0; e < 64; ++e) sv[h * 64 + e] = e < vh[h] ? sv[h * 64 + e] : -INFINITY;
            }
          }
        }
        if (!kExact && n < C::kWGs) {
          if (n == 0) look_at_first(ragged_tag, sv, vh);
          else learn_ref();
          if (exact) return;  // the variant with the turns takes the tile
        }
        // S is in registers: the Q K^T of tile g+2 may overwrite the buffer
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(s_free + wg);

        float alpha = 1.0f;
        if (kExact) {
          const float mx = row_max(sv, vh);
          // ---- my turn to look at / move the row's reference maximum (strictly in tile order) ----
          if (n > 0) take_turn();
          alpha = move_ref(mx);
          if (n == 0 && m_ref == -INFINITY) ref[row] = m_ref;
          if (n + 1 < n_tiles) give_turn();
        }

        // exponentials of keys [64h, 64h+64) -> packed bf16 columns [32h, 32h+32) of the P buffer
        uint32_t pk[64];
        const float2 sc2 = make_float2(p.scale_log2, p.scale_log2), nm2 = make_float2(-m_ref, -m_ref);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float* svh = sv + h * 64;
          uint32_t* pkh = pk + h * 32;
          if (vh[h] > 0) {  // then the row has a finite reference
#pragma unroll
            for (int e = 0; e < 32; ++e) {
              const float2 x = ffma2(make_float2(svh[2 * e], svh[2 * e + 1]), sc2, nm2);
              constexpr int kPoly = SPARSP_TUNE_POLY;
              const float2 pp = (kPoly > 0 && (e % (kPoly > 0 ? kPoly : 1)) == 1)
                                    ? exp2_poly2<kRagged || kExact, !kExact>(x, &i_max)
                                    : make_float2(ex2(x.x), ex2(x.y));
              const __nv_bfloat162 h2 = __floats2bfloat162_rn(pp.x, pp.y);
              pkh[e] = *reinterpret_cast<const uint32_t*>(&h2);
            }
            if (kRagged && vh[h] < 64) {
              // columns past the end of the sequence: exactly zero in P (the polynomial path returns
              // 2^-126 for them, which the row sum may keep)
#pragma unroll
              for (int e = 0; e < 32; ++e)
                pkh[e] = 2 * e + 1 < vh[h] ? pkh[e] : (2 * e < vh[h] ? (pkh[e] & 0xffffu) : 0u);
            }
          } else {
#pragma unroll
            for (int e = 0; e < 32; ++e) pkh[e] = 0u;
          }
        }
        // the P buffer was last read by the P V of tile g-1
        if (g >= 1) {
          mbar_wait_bounded_inline(o_full + ((g - 1) & 3), ((g - 1) >> 2) & 1, s_abort, 34 + wg, p.wait_limit);
          tc_fence_after();
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_st16(tP + c * 16, pk + c * 16);
        if (kExact) rescale(alpha, n);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full + wg);
        round ^= 1u;
      };

      // One tile of this warpgroup.  kRagged = the sequence ends inside the tile (possible only for the item's last
      // one), or (K / V source) the reference comes from the first tile and this is it: that variant carries the column
      // masking; kExact: the one with the turns.  The common variant stays small.
      auto do_tile = [&](auto ragged_tag, auto exact_tag, const int n) {
        constexpr bool kRagged = decltype(ragged_tag)::value;
        // kept / valid key columns of each 64-column half of the tile (warp-uniform), as the list builder left them
        int vh[2];
        if (C::kStacked) {
          // both entries at once; an odd list ends with one that nobody keeps
          if constexpr (kPacked) {
            const uint2 v = reinterpret_cast<const uint2*>(ent)[n];
            vh[0] = (v.x >> (E::kFlagShift + rh)) & 1u ? 64 : 0;
            vh[1] = (v.y >> (E::kFlagShift + rh)) & 1u ? 64 : 0;
          } else {
            const uint32_t v = reinterpret_cast<const uint32_t*>(ent)[n] >> (E::kFlagShift + rh);
            vh[0] = v & 1u ? 64 : 0;
            vh[1] = v & 0x10000u ? 64 : 0;
          }
        } else {
          vh[0] = vh[1] = 64;
        }
        if (kRagged && item_ragged && n == n_tiles - 1) {
          // the list's last entry is the block in which the sequence ends
          const int valid = (int)(p.N - (int64_t)(p.NB - 1) * BLK);
          if (C::kStacked) {
            if (n_ent & 1) vh[0] = min(vh[0], valid);
            else vh[1] = min(vh[1], valid);
          } else {
            vh[0] = min(valid, 64);
            vh[1] = max(valid - 64, 0);
          }
        }
        mbar_wait_bounded_inline(s_full + wg, round, s_abort, 30 + wg, p.wait_limit);
        tc_fence_after();
        if constexpr (C::kInPlaceP) in_place_tile(ragged_tag, exact_tag, n, vh);
        else own_buffer_tile(ragged_tag, exact_tag, n, vh);
      };
      // (nothing to learn: the barriers keep step)
      if (exact && first == 0 && lane == 0) mbar_arrive(ref_ready + (i & 3));
      int n = first;
      // the list builder puts the sequence's last block (the only one that can be ragged) into the last tile
      const int n_rag = item_ragged ? n_tiles - 1 : -1;
      if (!exact) {
        for (; n < n_tiles; n += C::kWGs) {
          if (n == n_rag || (!kPacked && ref_of == kRefFirst && n < C::kWGs))
            do_tile(std::true_type{}, std::false_type{}, n);
          else
            do_tile(std::false_type{}, std::false_type{}, n);
          if (exact) break;  // what the first tile says
        }
      }
      if (exact)
        for (; n < n_tiles; n += C::kWGs) do_tile(std::true_type{}, std::true_type{}, n);

      g0 += n_tiles;
      w0 = (w0 + n_tiles) % C::kWGs;
      // ---- item epilogue: the warpgroup of the item's last tile writes the rows, the other one goes on ----
      const int last = g0 - 1;
      if ((w0 == 0 ? C::kWGs - 1 : w0 - 1) != wg) {
        if (__any_sync(0xffffffffu, !exact && !(i_max <= kMaxExponent)) && lane == 0) s_failed[buf] = 1;
        __syncwarp();
        if (hd.y & kHeadMeet) {
          if (lane == 0) mbar_arrive(placed);
          mbar_wait_bounded_inline(placed, (hd.y >> kHeadMeetParityShift) & 1, s_abort, 45, p.wait_limit);
        }
        if (lane == 0) mbar_arrive(list_free + buf);
      } else {
        const int qb = C::kStacked && rh ? (int)((uint32_t)hd.z >> 16) : hd.z & 0xffff;
        // (a block that keeps nothing is stacked with one that does: other warps write its rows)
        const bool none = qb == 0xffff || ((hd.y >> (kHeadNoneShift + (C::kStacked ? rh : 0))) & 1);
        int64_t tok = none ? p.N : (int64_t)qb * BLK + (C::kStacked ? (row & 63) : row);
        __nv_bfloat16* orow = p.O + (int64_t)hd.w * p.sB + (int64_t)(hd.x - hd.w * p.H) * p.sH + tok * p.sT;
        float* lrow = p.lse ? p.lse + (int64_t)hd.x * p.N + tok : nullptr;
        // a thread's row is 2 D contiguous bytes but the rows of a warp are sT elements apart, so every
        // store instruction touches 32 lines: 32-byte stores (when the layout allows) halve their number
        int wide = ((reinterpret_cast<uintptr_t>(orow) | (uintptr_t)(p.sT * 2)) & 31) == 0, mine_to_write = tok < p.N;
        // (worked out while the last P V runs, not behind it)
        asm volatile("" : "+l"(orow), "+l"(lrow), "+r"(wide), "+r"(mine_to_write));
        mbar_wait_bounded_inline(o_full + (last & 3), (last >> 2) & 1, s_abort, 40, p.wait_limit);
        tc_fence_after();
        uint32_t o[D + 1];  // the row's accumulator and its sum
        tmem_ld1(tmem_base + C::kColL + lane_off, o + D);
#pragma unroll
        for (int c = 0; c < D / 32; ++c) tmem_ld32(tO + c * 32, o + c * 32);
        tmem_ld_wait(o);
        // the accumulator is in registers: the next item's first P V may overwrite it
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(o_drained);
        const float l = __uint_as_float(o[D]);
        // (an ordinary item asks one question here)
        const float safe = ref_of == kRefZero ? kSafeSumZero : kSafeSumFirst;
        const bool asks = !exact && mine_to_write && !(i_max <= kMaxExponent && l >= kMinSum && l <= safe);
        if (__any_sync(0xffffffffu, asks) || (hd.y & kHeadMeet)) {
          bool failed = asks && !(i_max <= kMaxExponent && l >= kMinSum && l <= kMaxSum);
          if (asks) {
            float most = 0.0f;  // has a column run out of fp32?
#pragma unroll
            for (int e = 0; e < D; e += 2) most = max_abs3(__uint_as_float(o[e]), __uint_as_float(o[e + 1]), most);
            failed = failed || !(most < INFINITY);
          }
          if (__any_sync(0xffffffffu, failed) && lane == 0) s_failed[buf] = 1;
          __syncwarp();
          if (hd.y & kHeadMeet) {  // (in place, the rows of an item that is to be computed again are still its queries)
            if (lane == 0) mbar_arrive(placed);
            mbar_wait_bounded_inline(placed, (hd.y >> kHeadMeetParityShift) & 1, s_abort, 45, p.wait_limit);
            if (s_failed[buf]) mine_to_write = 0;
          }
        }
        if (lane == 0) mbar_arrive(list_free + buf);
        const float inv_l = l > 0.0f ? 1.0f / l : 0.0f;
        if (mine_to_write) {
#pragma unroll
          for (int v = 0; v < D / 16; ++v) {
            uint32_t w[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(o[v * 16 + 2 * e]) * inv_l,
                                                              __uint_as_float(o[v * 16 + 2 * e + 1]) * inv_l);
              w[e] = *reinterpret_cast<const uint32_t*>(&h2);
            }
            if (wide) {
              asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(orow + v * 16), "r"(w[0]),
                           "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                           : "memory");
            } else {
              *reinterpret_cast<uint4*>(orow + v * 16) = make_uint4(w[0], w[1], w[2], w[3]);
              *reinterpret_cast<uint4*>(orow + v * 16 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
            }
          }
        }
        if (lrow && mine_to_write)  // (a score that is no number makes the row's sum none, or infinite)
          *lrow = !(l < INFINITY) ? NAN : l > 0.0f ? (m_ref + log2f(l)) * 0.6931471805599453f : -INFINITY;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, kTmemCols);
  if (tid == 0) report_abort(s_abort, p.status);
}

// ------------------------------------------------------------------------------------------------
// Preparation of an attention call: a CTA per (batch, head) fixes its work items and, packed source, another one its
// table of packed slots.  A query block that keeps nothing never becomes a work item.
//
// Block 64: which two query blocks share a Q tile.  K / V source: blocks i and i+D are paired in stripes (i mod 2D <
// D), leftovers pair up consecutively; the offset D in 1..n/2 that maximises the summed overlap |M[i] & M[i+D]| of the
// kept lists is chosen per (batch, head) -- video attention is multi-diagonal, so the best partner of a block is
// typically the same position a fixed number of blocks away; the more two stacked blocks share, the less of a 128-row
// tile's work is masked away.
// Packed source: neighbours in the consumer's ascending list of blocks (D = 1), so that a row's result depends on its
// neighbour's list at most, not on what the consumer's other blocks keep.
// (Mask rows in shared memory have a pitch of an odd number of 16-byte units, which are read whole: the threads'
// offsets differ by one row, an even pitch would put many of them on the same banks.)
// Items of one (batch, head) are handed out longest list first: the items still running when the queue runs dry are
// then the short ones, which matters when list lengths vary (threshold selection, unions of two stacked blocks).  Key =
// (list length << 10) | (1023 - index): up to kPrepThreads / 2 items of equal length keep their index order, more of
// them are in any order.
// Latency-bound integer work, so what matters is how many loads and barriers wait for each other: rows are counted by a
// warp each with eight in flight, items are put in order without rounds, offsets are scored by all threads, and slots
// have CTAs of their own and no shared-memory atomics.  One hop of 40 heads x 591 blocks, 8 ranks 5.9 us (23 with 256
// threads, a thread per row, a bitonic sort for any number and the slots behind the items), 24 x 384 stacked blocks
// 15.5, 2 x 64 4.5 (attention calls 72 -> 66-74, 617 -> 594 and 21.2 -> 19.4 us).
// ------------------------------------------------------------------------------------------------
constexpr int kPrepThreads = 512;
constexpr int kPairSample = 8;

struct PrepParams {
  const uint32_t* mask;
  int32_t* pairs;
  int32_t* n_items;
  int32_t* work_counter;
  int BH, H, NB, Wd, b;
  // packed source only
  const int32_t* rank;
  const uint32_t* U;
  const int64_t* seg_off;
  const int64_t* seg_total;
  const int64_t* dst_base;
  int64_t tile_bytes;
  int32_t* slot;
  int64_t* tile_base;
  int P, consumer;
};

// Sorts n keys (n a power of two; up to kPrepThreads / 2, or kMany: 1024) in shared memory by length, the longest
// first; all threads call it.
template <bool kMany>
__device__ __forceinline__ void sort_keys_descending(uint32_t* keys, int n) {
  if constexpr (!kMany) {
    // Few keys: a key's place is the number of larger ones, counted by two threads.  No rounds that wait for each
    // other.
    const int k = threadIdx.x >> 1;
    const uint32_t key = k < n ? keys[k] : 0u;
    int place = 0;
    if (key != 0u)
      for (int j = threadIdx.x & 1; j < n; j += 2) place += keys[j] > key ? 1 : 0;
    place += __shfl_xor_sync(0xffffffffu, place, 1);
    __syncthreads();
    if (k < n && (threadIdx.x & 1) == 0) keys[k] = 0u;
    __syncthreads();
    if (key != 0u && (threadIdx.x & 1) == 0) keys[place] = key;
    __syncthreads();
  } else {
    // Many keys: a place for every length, by counting; equal lengths in any order, a warp's together.
    constexpr int kLens = kMaxBlocks + 1, kPer = (kLens + kPrepThreads - 1) / kPrepThreads, kWarps = kPrepThreads / 32;
    constexpr int kKeys = kMaxBlocks / kPrepThreads;
    // place kLens - 1 - length: keys of that length, then where they begin
    __shared__ int at_s[kPer * kPrepThreads], sum_s[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int t = 0; t < kPer; ++t) at_s[threadIdx.x + t * kPrepThreads] = 0;
    uint32_t key[kKeys], peers[kKeys];
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kKeys; ++t) {
      const int i = threadIdx.x + t * kPrepThreads;
      key[t] = i < n ? keys[i] : 0u;
      peers[t] = __match_any_sync(0xffffffffu, key[t] >> 10);
      if (lane == __ffs(peers[t]) - 1) atomicAdd(&at_s[kLens - 1 - (key[t] >> 10)], __popc(peers[t]));
    }
    __syncthreads();
    int mine[kPer], sum = 0;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      mine[t] = at_s[threadIdx.x * kPer + t];
      sum += mine[t];
    }
    int incl = sum;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, s);
      if (lane >= s) incl += v;
    }
    if (lane == 31) sum_s[warp] = incl;
    __syncthreads();
    int begin = incl - sum;
#pragma unroll
    for (int k = 0; k < kWarps; ++k) begin += k < warp ? sum_s[k] : 0;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      at_s[threadIdx.x * kPer + t] = begin;
      begin += mine[t];
    }
    __syncthreads();
#pragma unroll
    for (int t = 0; t < kKeys; ++t) {
      const int leader = __ffs(peers[t]) - 1;
      int place = 0;
      if (lane == leader) place = atomicAdd(&at_s[kLens - 1 - (key[t] >> 10)], __popc(peers[t]));
      place = __shfl_sync(0xffffffffu, place, leader) + __popc(peers[t] & ((1u << lane) - 1u));
      if (place < n) keys[place] = key[t];
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int next_pow2(int n) {
  int v = 1;
  while (v < n) v <<= 1;
  return v;
}

// Work items of one (batch, head) among the n query blocks list[0..n) (packed source; NULL: all blocks, K / V source);
// returns their number.
template <bool kStacked, bool kMany>
__device__ __forceinline__ int make_items(const PrepParams& p, int bh, const uint16_t* list, int n,
                                          unsigned char* smem_raw) {
  __shared__ uint32_t s_keys[kMaxBlocks];
  __shared__ uint32_t s_pair[kMaxBlocks / 2];  // positions of an item's two blocks, (second or 0xffff) << 16 | first
  __shared__ unsigned int s_score[kMaxBlocks / 2];
  __shared__ unsigned int s_best;              // (score << 10) | (1023 - D): max = best score, smallest D
  const uint32_t* rows = p.mask + (int64_t)bh * p.NB * p.Wd;
  auto block = [&](int pos) -> int { return list ? list[pos] : pos; };
  int n_keys;
  bool live = false;  // any of my keys is an item's
  if constexpr (kStacked) {
    uint32_t* m = reinterpret_cast<uint32_t*>(smem_raw);  // [n][pitch], zeros behind a row's words
    const uint4* m4 = reinterpret_cast<const uint4*>(smem_raw);
    const int Wd = p.Wd, units = (Wd + 3) / 4, pitch4 = units | 1, pitch = 4 * pitch4;
    if (threadIdx.x == 0) s_best = 1023u - 1u;  // default D = 1
    for (int i = threadIdx.x; i < n; i += kPrepThreads)
      for (int w = Wd; w < 4 * units; ++w) m[i * pitch + w] = 0u;
    auto read = [&](auto in_flight) {
      constexpr int kFlight = decltype(in_flight)::value;
      for (int idx0 = threadIdx.x; idx0 < n * Wd; idx0 += kFlight * kPrepThreads) {
        uint32_t v[kFlight];
        int at[kFlight];
#pragma unroll
        for (int u = 0; u < kFlight; ++u) {
          const int idx = idx0 + u * kPrepThreads, i = idx / Wd, w = idx - i * Wd;
          at[u] = idx < n * Wd ? i * pitch + w : -1;
          v[u] = at[u] >= 0 ? rows[(int64_t)block(i) * Wd + w] : 0u;
        }
#pragma unroll
        for (int u = 0; u < kFlight; ++u)
          if (at[u] >= 0) m[at[u]] = v[u];
      }
    };
    if (n * Wd <= kPrepThreads) read(std::integral_constant<int, 1>{});
    else read(std::integral_constant<int, 8>{});
    // bits that two rows share, or that either has
    auto common = [&](int a, int b2, bool either) {
      int bits = 0;
      for (int u = 0; u < units; ++u) {
        const uint4 x = m4[a * pitch4 + u], y = m4[b2 * pitch4 + u];
        bits += either ? __popc(x.x | y.x) + __popc(x.y | y.y) + __popc(x.z | y.z) + __popc(x.w | y.w)
                       : __popc(x.x & y.x) + __popc(x.y & y.y) + __popc(x.z & y.z) + __popc(x.w & y.w);
      }
      return bits;
    };
    __syncthreads();
    if (!list && n > 1) {
      const int n_off = n / 2, parts = max(1, kPrepThreads / n_off);  // threads per offset
      for (int t = threadIdx.x; t < n_off; t += kPrepThreads) s_score[t] = 0u;
      __syncthreads();
      for (int t = threadIdx.x; t < n_off * parts; t += kPrepThreads) {
        const int part = t / n_off, d = 1 + t - part * n_off;
        unsigned int score = 0;
        // every kPairSample-th row is enough to rank offsets
        for (int i = part * kPairSample; i + d < n; i += kPairSample * parts)
          score += (unsigned int)common(i, i + d, false);
        atomicAdd(&s_score[d - 1], score);
      }
      __syncthreads();
      for (int t = threadIdx.x; t < n_off; t += kPrepThreads)
        atomicMax(&s_best, (s_score[t] << 10) | (unsigned int)(1023 - (t + 1)));
    }
    __syncthreads();
    const int D = 1023 - (int)(s_best & 1023u);
    // stripes: positions with (i mod 2D) < D pair with i + D; the positions of the last partial stripe that have
    // no partner form one consecutive run and pair up as neighbours
    const int full = n / (2 * D), R = n % (2 * D);
    const int np_last = max(R - D, 0), lo_end = min(R, D);
    for (int i = threadIdx.x; i < n; i += kPrepThreads) {
      const int st = i / (2 * D), pos = i % (2 * D);
      if (st < full) {
        if (pos < D) s_pair[st * D + pos] = (uint32_t)(i + D) << 16 | (uint32_t)i;
      } else if (pos < np_last) {
        s_pair[full * D + pos] = (uint32_t)(i + D) << 16 | (uint32_t)i;
      } else if (pos < lo_end) {
        const int k = pos - np_last, n_left = lo_end - np_last;
        if ((k & 1) == 0)
          s_pair[full * D + np_last + k / 2] = (k + 1 < n_left ? (uint32_t)(i + 1) : 0xffffu) << 16 | (uint32_t)i;
      }
    }
    __syncthreads();
    n_keys = (n + 1) / 2;
    for (int c = threadIdx.x; c < next_pow2(n_keys); c += kPrepThreads) {
      uint32_t key = 0;
      if (c < n_keys) {
        const int a = (int)(s_pair[c] & 0xffffu), b2 = (int)(s_pair[c] >> 16);
        const int len = common(a, b2 != 0xffff ? b2 : a, true);
        key = ((uint32_t)len << 10) | (uint32_t)(1023 - c);
      }
      s_keys[c] = key;
      live = live || (key >> 10) != 0u;
    }
  } else {
    // a warp per row, kPrepRows rows of loads in flight
    n_keys = n;
    constexpr int kPrepRows = 8, kWarps = kPrepThreads / 32;
    const int lane = threadIdx.x & 31, n_pow2 = next_pow2(n_keys);
    for (int i0 = threadIdx.x >> 5; i0 < n_pow2; i0 += kWarps * kPrepRows) {
      uint32_t v[kPrepRows];
#pragma unroll
      for (int k = 0; k < kPrepRows; ++k) {
        const int i = i0 + k * kWarps;
        v[k] = i < n && lane < p.Wd ? rows[(int64_t)block(i) * p.Wd + lane] : 0u;
      }
#pragma unroll
      for (int k = 0; k < kPrepRows; ++k) {
        const int i = i0 + k * kWarps, len = __reduce_add_sync(0xffffffffu, __popc(v[k]));
        if (lane == 0 && i < n_pow2) s_keys[i] = i < n ? ((uint32_t)len << 10) | (uint32_t)(1023 - i) : 0u;
        live = live || len > 0;
      }
    }
  }
  if (!__syncthreads_or(live)) return 0;
  sort_keys_descending<kMany>(s_keys, next_pow2(n_keys));
  int32_t* out = p.pairs + (int64_t)bh * (2 * ((p.NB + 1) / 2));
  int n_live = 0;
  for (int x0 = 0; x0 < n_keys; x0 += kPrepThreads) {
    const int x = x0 + (int)threadIdx.x;
    const bool is_item = x < n_keys && (s_keys[x] >> 10) != 0u;
    if (is_item) {
      const int c = 1023 - (int)(s_keys[x] & 1023u);
      if (kStacked) {
        const int a = (int)(s_pair[c] & 0xffffu), b2 = (int)(s_pair[c] >> 16);
        out[2 * x] = block(a);
        out[2 * x + 1] = b2 != 0xffff ? block(b2) : -1;
      } else {
        out[x] = block(c);
      }
    }
    n_live += __syncthreads_count(is_item);
  }
  return n_live;
}

// slot[bh][j] = entry index of block j inside the consumer's packed buffer (pack order: producer ascending,
// head ascending, block ascending), for every block of the consumer's union that another rank owns; -1 elsewhere.
// First the entry index of every word of every producer's set, a warp per producer; then a thread per block.
__device__ __forceinline__ void make_slots(const PrepParams& p, int bh) {
  __shared__ uint32_t set_s[kMaxRanks * kMaxWords];
  __shared__ int32_t at_s[kMaxRanks * kMaxWords];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int bb = bh / p.H, h = bh % p.H;
  const int64_t br = (int64_t)bb * p.P + p.consumer;
  const uint32_t u = lane < p.Wd ? p.U[(br * p.H + h) * p.Wd + lane] : 0u;
  for (int prod = warp; prod < p.P; prod += kPrepThreads / 32) {
    const int64_t first = p.seg_off[(br * p.P + prod) * p.H + h];
    uint32_t set = 0;
#pragma unroll 8
    for (int w = 0; w < p.Wd; ++w) {
      const int j = w * 32 + lane;
      const uint32_t word = __ballot_sync(0xffffffffu, j < p.NB && p.rank[j] == prod);
      if (lane == w) set = word & u;
    }
    int total;
    const int below = bits_below(set, lane, &total);
    if (lane < p.Wd) {
      set_s[prod * p.Wd + lane] = set;
      at_s[prod * p.Wd + lane] = (int)first + below;
    }
  }
  __syncthreads();
  int32_t* out = p.slot + (int64_t)bh * p.NB;
  for (int j = threadIdx.x; j < p.NB; j += kPrepThreads) {
    const int prod = p.rank[j], bit = j & 31;
    int slot = -1;
    if ((unsigned)prod < (unsigned)p.P && prod != p.consumer) {
      const uint32_t set = set_s[prod * p.Wd + (j >> 5)];
      if ((set >> bit) & 1u) slot = at_s[prod * p.Wd + (j >> 5)] + __popc(set & ((1u << bit) - 1u));
    }
    out[j] = slot;
  }
}

// (An instance for each form, because the launch waits for the code it is given: with all of it in one, layers of a few
// thousand tokens took 6 us longer.)
template <bool kPacked, bool kStacked, bool kMany>
__global__ void __launch_bounds__(kPrepThreads) attn_prep_kernel(const PrepParams p) {
  enter_grid();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.work_counter = 0;  // the attention kernel's work queue
  const int bh = blockIdx.x;
  if (kPacked && bh >= p.BH) {
    make_slots(p, bh - p.BH);
    return;
  }
  int n_live;
  if (kPacked) {
    __shared__ uint32_t s_words[kMaxWords];
    __shared__ uint16_t s_list[kMaxBlocks];
    rank_words(p.rank, p.NB, p.consumer, s_words);
    const int n = list_blocks(s_words, p.NB, s_list);
    n_live = make_items<kStacked, kMany>(p, bh, s_list, n, smem_raw);
    if (bh % p.H == 0 && warp == 0) {  // first tile of the consumer's buffer for this batch item
      const int64_t br = (int64_t)(bh / p.H) * p.P + p.consumer;
      int64_t first = 0;
      if (p.dst_base) {
        first = p.dst_base[br] / p.tile_bytes;
      } else {
        for (int64_t t = lane; t < br; t += 32) first += 2 * p.seg_total[t];
#pragma unroll
        for (int s = 16; s >= 1; s >>= 1) first += __shfl_xor_sync(0xffffffffu, first, s);
      }
      if (lane == 0) p.tile_base[bh / p.H] = first;
    }
  } else {
    n_live = make_items<kStacked, kMany>(p, bh, nullptr, p.NB, smem_raw);
  }
  if (threadIdx.x == 0) p.n_items[bh] = n_live;
}

// ------------------------------------------------------------------------------------------------
// host side: tensor maps and launch
// ------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// bf16 tensor viewed as (d, N, H, B) with a box of (d, rows, 1, 1), or of (64, rows, 1, 1) and 128-byte swizzle.
// A dimension of extent 1 takes a stride of its own choice (whatever the caller has there is never used).
int make_tile_tmap(CUtensorMap* out, const void* base, const sparsp_shape& s, const Geometry& g, int rows,
                   bool swizzled) {
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return SPARSP_ERR_CUDA;
  }
  cuuint64_t dims[4] = {(cuuint64_t)g.d, (cuuint64_t)g.N, (cuuint64_t)g.H, (cuuint64_t)g.B};
  const int64_t head_stride = g.H > 1 ? s.stride_head : s.stride_token;
  const int64_t batch_stride = g.B > 1 ? s.stride_batch : s.stride_token;
  cuuint64_t strides[3] = {(cuuint64_t)s.stride_token * 2, (cuuint64_t)head_stride * 2, (cuuint64_t)batch_stride * 2};
  cuuint32_t box[4] = {swizzled ? 64u : (cuuint32_t)g.d, (cuuint32_t)rows, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, swizzled ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed with %d", (int)r);
    return SPARSP_ERR_CUDA;
  }
  return SPARSP_OK;
}

// Packed buffer viewed as a sequence of (block x d) bf16 tiles: dims (d, block, n_tiles, 1).
static int make_packed_tmap(CUtensorMap* out, const void* packed, int64_t capacity_bytes, const Geometry& g) {
  EncodeTiledFn enc = get_encode_fn();
  if (!enc) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return SPARSP_ERR_CUDA;
  }
  const int64_t tile_bytes = (int64_t)g.b * g.d * 2;
  const int64_t n_tiles = capacity_bytes / tile_bytes;
  if (n_tiles < 1 || n_tiles > 0x7fffffff) {
    set_error("packed buffer holds %lld tiles: outside 1..2^31-1", (long long)n_tiles);
    return SPARSP_ERR_INVALID_ARG;
  }
  cuuint64_t dims[4] = {(cuuint64_t)g.d, (cuuint64_t)g.b, (cuuint64_t)n_tiles, 1};
  cuuint64_t strides[3] = {(cuuint64_t)g.d * 2, (cuuint64_t)tile_bytes, (cuuint64_t)(tile_bytes * n_tiles)};
  cuuint32_t box[4] = {64, (cuuint32_t)g.b, 1, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = enc(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(packed), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled (packed) failed with %d", (int)r);
    return SPARSP_ERR_CUDA;
  }
  return SPARSP_OK;
}

template <int D, int BLK, Source kSource>
static int launch_attn_t(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, const void* V,
                         const void* packed, int64_t packed_capacity, const AttnParams& p, cudaStream_t st) {
  CUtensorMap tq, tk, tv, tp;
  int rc;
  if ((rc = make_tile_tmap(&tq, Q, s, g, BLK, true)) != SPARSP_OK) return rc;
  if ((rc = make_tile_tmap(&tk, K, s, g, BLK, true)) != SPARSP_OK) return rc;
  if ((rc = make_tile_tmap(&tv, V, s, g, BLK, true)) != SPARSP_OK) return rc;
  if (kSource == Source::kPacked || kSource == Source::kPackedDirect) {
    if ((rc = make_packed_tmap(&tp, packed, packed_capacity, g)) != SPARSP_OK) return rc;
  } else {
    tp = tk;  // never used
  }
  auto kern = attn_fwd_kernel<D, BLK, kSource>;
  constexpr bool kNoQueue = kSource == Source::kPackedDirect || kSource == Source::kDirect;
  const int smem = kNoQueue ? AttnCfg<D, BLK>::kDynamicDirect : AttnCfg<D, BLK>::kDynamic;
  SPARSP_CUDA_OK(ensure_dynamic_smem((const void*)kern, smem));
  // work item = one 128-row Q tile (a 128-token block, a pair of 64-token blocks, or one of them); one persistent CTA
  // per SM
  const int64_t most = (int64_t)g.B * g.H * (BLK == 128 || kSource == Source::kDirect ? g.NB : (g.NB + 1) / 2);
  int sms = 0;
  SPARSP_CUDA_OK(sm_count(&sms));
  const unsigned grid = (unsigned)std::min<int64_t>(most, sms);
  // The warpgroups share out the registers that the block is launched with; should a build of the kernel be given
  // fewer, some of them would wait for good.
  constexpr int kSoftmax = AttnCfg<D, BLK>::kWGs * AttnCfg<D, BLK>::kRegsSoftmax;
  constexpr int kShared = 128 * (SPARSP_REGS_UTILITY + SPARSP_REGS_UTILITY2 + kSoftmax);
  static std::atomic<int> launched_with{0};
  if (launched_with.load(std::memory_order_relaxed) < kShared) {
    cudaFuncAttributes attr;
    SPARSP_CUDA_OK(cudaFuncGetAttributes(&attr, (const void*)kern));
    launched_with.store(attr.numRegs * AttnCfg<D, BLK>::kThreads, std::memory_order_relaxed);
    if (attr.numRegs * AttnCfg<D, BLK>::kThreads < kShared) {
      set_error("the attention kernel was built with %d registers a thread: too few to share out", attr.numRegs);
      return SPARSP_ERR_UNSUPPORTED;
    }
  }
  SPARSP_CUDA_OK(launch_kernel(kern, grid, AttnCfg<D, BLK>::kThreads, smem, st, tq, tk, tv, tp, p));
  return SPARSP_OK;
}

template <Source kSource>
static int launch_attn_common(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, const void* V,
                              const void* packed, int64_t packed_capacity, AttnParams p, float scale, void* O,
                              float* lse, char* ws, const WsLayout& L, cudaStream_t st) {
  p.O = (__nv_bfloat16*)O;
  p.lse = lse;
  p.in_place = O == Q;
  p.status = (int32_t*)(ws + L.status);
  p.work_counter = p.status + kWorkCounterWord;
  p.N = g.N;
  p.sB = s.stride_batch;
  p.sH = s.stride_head;
  p.sT = s.stride_token;
  p.BH = g.B * g.H;
  p.H = g.H;
  p.NB = g.NB;
  p.Wd = g.Wd;
  const float sc = scale > 0.0f ? scale : 1.0f / sqrtf((float)g.d);
  p.scale_log2 = sc * 1.4426950408889634f;
  p.wait_limit = 200000000LL;  // about 0.1 s of SM clocks
  if (g.d == 64 && g.b == 64) return launch_attn_t<64, 64, kSource>(s, g, Q, K, V, packed, packed_capacity, p, st);
  if (g.d == 64 && g.b == 128) return launch_attn_t<64, 128, kSource>(s, g, Q, K, V, packed, packed_capacity, p, st);
  if (g.d == 128 && g.b == 64) return launch_attn_t<128, 64, kSource>(s, g, Q, K, V, packed, packed_capacity, p, st);
  return launch_attn_t<128, 128, kSource>(s, g, Q, K, V, packed, packed_capacity, p, st);
}

template <bool kPacked>
static int launch_prep(const Geometry& g, const PrepParams& p, cudaStream_t st) {
  const bool many = (g.b == 64 ? (g.NB + 1) / 2 : g.NB) > kPrepThreads / 2;
  auto kern = g.b == 64 ? (many ? attn_prep_kernel<kPacked, true, true> : attn_prep_kernel<kPacked, true, false>)
                        : (many ? attn_prep_kernel<kPacked, false, true> : attn_prep_kernel<kPacked, false, false>);
  const int smem = g.b == 64 ? g.NB * (((g.Wd + 3) / 4) | 1) * 16 : 0;
  SPARSP_CUDA_OK(ensure_dynamic_smem((const void*)kern, smem));
  SPARSP_CUDA_OK(launch_kernel(kern, (unsigned)(kPacked ? 2 * p.BH : p.BH), kPrepThreads, smem, st, p));
  return SPARSP_OK;
}

static PrepParams prep_params(const Geometry& g, const uint32_t* mask, char* ws, const WsLayout& L) {
  PrepParams p = {};
  p.mask = mask;
  p.pairs = (int32_t*)(ws + L.pairs);
  p.n_items = (int32_t*)(ws + L.n_items);
  p.work_counter = (int32_t*)(ws + L.status) + kWorkCounterWord;
  p.BH = g.B * g.H;
  p.H = g.H;
  p.NB = g.NB;
  p.Wd = g.Wd;
  p.b = g.b;
  return p;
}

int launch_attn(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, const void* V,
                const uint32_t* mask, float scale, void* O, float* lse, char* ws, const WsLayout& L,
                cudaStream_t st) {
  AttnParams p = {};
  p.mask = mask;
  // So few query blocks need no queue and no launch that fills it.  64-token blocks: one an SM; an item is then done
  // sooner with its own list than with the union of two (us a call with the launch that makes items / without it: 2
  // heads x 64 blocks of 64 x 64, 16 kept 14.9 / 11.5, stacked 19.4).  More of them have to share Q tiles where
  // neighbours keep the same blocks: 2 x 100 of 64 x 128, a quarter kept in windows 22.5 with the queue, 30.9
  // unstacked, all kept 50 / 83 (threshold lists, whose unions are long, would gain: 2 x 120 77 / 52).  128-token
  // blocks: two an SM; every CTA puts them in order for itself and takes one from the front and one from behind (7 x 21
  // of 64 x 128 15.7 / 10.4, 2 x 148 of 128 x 128, 15 % kept 58.5 / 52.9, threshold lists 67 / 54; up to three an SM
  // 0.90 to 1.10 times as fast, up to four 0.80 to 1.04).  An instance of the kernel of its own, because the question
  // inside the queue's made 64-token blocks 1-2 % slower.
  int sms = 0;
  SPARSP_CUDA_OK(sm_count(&sms));
  if ((int64_t)g.B * g.H * g.NB <= std::min((g.b == 64 ? 1 : 2) * sms, kMaxDirect))
    return launch_attn_common<Source::kDirect>(s, g, Q, K, V, nullptr, 0, p, scale, O, lse, ws, L, st);
  const PrepParams pre = prep_params(g, mask, ws, L);
  const int rc = launch_prep<false>(g, pre, st);
  if (rc != SPARSP_OK) return rc;
  p.pairs = pre.pairs;
  p.n_items = pre.n_items;
  return launch_attn_common<Source::kQueue>(s, g, Q, K, V, nullptr, 0, p, scale, O, lse, ws, L, st);
}

// ------------------------------------------------------------------------------------------------
// Packed-source attention for one consumer rank: items are formed among the consumer's own query
// blocks, and every kept KV block the consumer does not own is read from the consumer's packed buffer.
// ------------------------------------------------------------------------------------------------
int launch_attn_packed(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, const void* V,
                       const uint32_t* mask, const int32_t* rank, int P, int consumer, const uint32_t* U,
                       const int64_t* seg_off, const int64_t* seg_total, const void* packed, int64_t capacity,
                       const int64_t* dst_base, float scale, void* O, float* lse, char* ws, const WsLayout& L,
                       cudaStream_t st) {
  AttnParams p = {};
  p.mask = mask;
  p.rank = rank;
  p.consumer = consumer;
  // Where the consumer has one item an SM at most, if it has its share of the blocks, neither their order nor a queue
  // matters, and the launch that makes them is left out: us a call over a whole buffer, with the launch / without, 1
  // head x 43 blocks, 5 ranks 18.5 / 16.4; an even share of 8 ranks, 15 % kept, 2 x 140 of 64 x 128 26.8 / 25.0, 4 x 97
  // of 64 x 128 21.2 / 19.1, 8 x 256 of 64 x 64 32.0 / 30.1, 7 x 146 of 128 x 128 33.2 / 30.1; a hop of 6 x 140 15.2 /
  // 13.0.  If the consumer has more than its share, the CTAs put its items in order for themselves, up to 1024 of them
  // (512 of heads of more than 512 blocks): 30 % of 8 x 128 of 64 x 128 42.9 / 42.0, with lists of unequal length 49.3
  // / 37.9, 30 % of 7 x 146 81.2 / 82.5 and 91.6 / 74.6, but all of short lists, 4 % kept, 8 x 128 39.9 / 43.3, 8 x 256
  // 64.8 / 76.6.  (In order of their numbers lists of unequal length took up to 1.7 times as long, half of 1 x 300 of
  // 128 x 128 75 / 110.  With two items an SM by an even share 4 x 300 of 128 x 128 34 / 44; 30 % of 2 x 1000 of 64 x
  // 128, whose rows are wide, 240 / 265.)
  int sms = 0;
  SPARSP_CUDA_OK(sm_count(&sms));
  const int64_t BH = (int64_t)g.B * g.H, share = (g.NB + P - 1) / P, per_item = 128 / g.b;
  const int64_t most = g.NB <= kPackedDirectBlocks ? kMaxPackedDirect : kMaxPackedDirect / 2;
  if (BH * ((share + per_item - 1) / per_item) <= sms && BH * ((g.NB + per_item - 1) / per_item) <= most) {
    p.P = P;
    p.U = U;
    p.seg_off = seg_off;
    p.seg_total = seg_total;
    p.dst_base = dst_base;
    p.tile_bytes = (int64_t)g.b * g.d * 2;
    return launch_attn_common<Source::kPackedDirect>(s, g, Q, K, V, packed, capacity, p, scale, O, lse, ws, L, st);
  }
  PrepParams pre = prep_params(g, mask, ws, L);
  pre.rank = rank;
  pre.U = U;
  pre.seg_off = seg_off;
  pre.seg_total = seg_total;
  pre.dst_base = dst_base;
  pre.tile_bytes = (int64_t)g.b * g.d * 2;
  pre.slot = (int32_t*)(ws + L.slot);
  pre.tile_base = (int64_t*)(ws + L.tile_base);
  pre.P = P;
  pre.consumer = consumer;
  const int rc = launch_prep<true>(g, pre, st);
  if (rc != SPARSP_OK) return rc;
  p.pairs = pre.pairs;
  p.n_items = pre.n_items;
  p.slot = pre.slot;
  p.tile_base = pre.tile_base;
  return launch_attn_common<Source::kPacked>(s, g, Q, K, V, packed, capacity, p, scale, O, lse, ws, L, st);
}

}  // namespace sparsp
