// Which work item a number of the attention kernel's queue stands for (K / V source), and which buffer a tile of an
// item lies in.  Plain integer code, apart from the kernel so that it can be run on a host as well.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define SPARSP_QUEUE_FN __device__ __forceinline__
#else
#define SPARSP_QUEUE_FN inline
#endif

namespace sparsp {

// Numbers run head by head, per_head to a head, of which only the first n_items[head] are items.  Returns the head of
// number `it` and its place *x among the head's items, or n_heads if there are no more.  A number behind a head's last
// item is exchanged: next(first number of the next head) hands out another one.  stop() ends the search without an
// item: the items' table is not written behind a head's last one, so nobody may look a place there up.
template <typename Next, typename Stop>
SPARSP_QUEUE_FN int find_item(int it, int per_head, int n_heads, const int32_t* n_items, Next next, Stop stop, int* x) {
  int head = it / per_head;
  *x = it - head * per_head;
  while (head < n_heads && *x >= n_items[head]) {
    if (stop()) return n_heads;
    it = next((head + 1) * per_head);
    head = it / per_head;
    *x = it - head * per_head;
  }
  return head;
}

// Which of the kRing + 1 shared buffers the next Q or K tile lies in, and the parity of its use: the producer and the Q
// K^T issuer both follow the same sequence of tiles.  A nibble per buffer, the next one lowest.
template <int kRing>
struct QKRing {
  uint32_t ring = kRing == 4 ? 0x3210u : 0x210u;
  uint32_t q = kRing;     // the item's Q tile (before the first item: the buffer that is not in the ring)
  uint32_t uses = 0u;     // bit b: parity of the uses of buffer b so far
  SPARSP_QUEUE_FN uint32_t use(uint32_t b) {  // parity of this use
    const uint32_t par = (uses >> b) & 1u;
    uses ^= 1u << b;
    return par;
  }
  SPARSP_QUEUE_FN uint32_t next_q() {
    const uint32_t b = ring & 15u;
    ring = (ring >> 4) | q << (4 * (kRing - 1));
    q = b;
    return b;
  }
  SPARSP_QUEUE_FN uint32_t next_k() {
    const uint32_t b = ring & 15u;
    ring = (ring >> 4) | b << (4 * (kRing - 1));
    return b;
  }
};

}  // namespace sparsp
