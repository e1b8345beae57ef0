// Which work item a number of the attention kernel's queue stands for (K / V source).  Plain integer code, apart from
// the kernel so that it can be run on a host as well.
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

}  // namespace sparsp
