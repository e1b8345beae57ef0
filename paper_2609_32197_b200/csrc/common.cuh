// Shared host-side plumbing of the SparSP library: geometry, error reporting, workspace layout.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cstdarg>
#include <cstdio>

#include "../../include/sparsp.h"

namespace sparsp {

constexpr int kMaxBlocks = 1024;  // NB limit (score rows are held in shared memory)
constexpr int kMaxRanks = 64;
constexpr int kStatusWords = 64;  // workspace header: word 0 = status code, 1.. = detail

struct Geometry {
  int64_t N;         // tokens
  int64_t n_video;   // video tokens
  int32_t NB;        // blocks
  int32_t Wd;        // mask words per row
  int32_t nb_cand;   // text-free blocks (top-k candidates); text blocks are NB - nb_cand tail blocks
  int32_t B, H, d, b;
};

struct WsLayout {
  int64_t status, pooled_q, pooled_k, scores, pairs, slot, tile_base, n_items, n_entries, entries, total;
};

void set_error(const char* fmt, ...);
int cuda_fail(cudaError_t e, const char* what);
extern std::atomic<int64_t> g_launches;
inline void count_launch(int n = 1) { g_launches.fetch_add(n, std::memory_order_relaxed); }

int make_geometry(const sparsp_shape* s, Geometry* g);
int check_strides(const sparsp_shape* s, const Geometry& g);
WsLayout make_layout(const Geometry& g, int n_ranks);

// Raises a kernel's dynamic shared-memory limit to at least `bytes` on the current device; remembers
// what was set per (kernel, device) so that the driver call is made only when the limit must grow.
cudaError_t ensure_dynamic_smem(const void* func, int bytes);

// Multiprocessors of the current device; asked of the driver once per device.
cudaError_t sm_count(int* sms);

// Launches a kernel that may start while the launches before it in the stream still run (programmatic stream
// serialisation): its CTAs take their places and set themselves up as soon as the previous kernel's have all started,
// and wait in enter_grid() before they touch memory, so that the latency of a launch is hidden behind the kernel before
// it. Every kernel launched here calls enter_grid() first thing, in every thread, or
// wait_previous_grids() where the next launch is to begin only as its CTAs end.
template <typename T>
struct same_type {
  using type = T;
};
// ... in clusters of `cluster` CTAs (the grid is a multiple of it)
template <typename... P>
inline cudaError_t launch_clusters(void (*kernel)(P...), dim3 grid, int cluster, int threads, size_t smem, cudaStream_t st,
                                   typename same_type<P>::type... args) {
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim = {(unsigned)cluster, 1, 1};
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, args...);
  if (e == cudaSuccess) count_launch();
  return e;
}
template <typename... P>
inline cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                                 typename same_type<P>::type... args) {
  return launch_clusters(kernel, grid, 1, threads, smem, st, args...);
}

#ifdef __CUDACC__
// Waits until all work before this launch has completed.  No thread returns or touches global memory before it.
// Pointers that the compiler may take for read-only are passed through it, so that no load through them can be moved
// ahead of the wait.
template <typename... P>
__device__ __forceinline__ void wait_previous_grids(P&... pointers) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  ((void)([](auto& p) { asm volatile("" : "+l"(p)::"memory"); }(pointers)), ...);
}
// First statement of a kernel started by launch_kernel: lets the next launch begin, then waits as above.
template <typename... P>
__device__ __forceinline__ void enter_grid(P&... pointers) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  wait_previous_grids(pointers...);
}
#endif

inline int64_t align_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

#define SPARSP_CUDA_OK(call)                              \
  do {                                                    \
    cudaError_t e__ = (call);                             \
    if (e__ != cudaSuccess) return cuda_fail(e__, #call); \
  } while (0)

int make_tile_tmap(CUtensorMap* out, const void* base, const sparsp_shape& s, const Geometry& g, int rows,
                   bool swizzled);

// launchers implemented in the kernel files -------------------------------------------------
int launch_pool(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, float* pq, float* pk, char* ws,
                const WsLayout& L, cudaStream_t st);
int launch_permute_tokens(const sparsp_shape& s, const Geometry& g, const void* X, void* Y,
                          const int32_t* block_of_slot, const int64_t* token_offset_of_slot, int inverse,
                          cudaStream_t st);
int launch_sharing(const Geometry& g, const uint32_t* mask, const int32_t* rank, int P, int64_t* hist,
                   cudaStream_t st);
int launch_score_cdf(const Geometry& g, const float* pq, const float* pk, float* scores, float tau, float scale,
                     uint32_t* mask, int32_t* kv_count, cudaStream_t st);
int launch_score_topk(const Geometry& g, const float* pq, const float* pk, float* scores, int topk,
                      uint32_t* mask, int32_t* kv_list, int32_t* kv_count, cudaStream_t st);
int launch_demand(const Geometry& g, const uint32_t* mask, const int32_t* rank_of_block, int P, int flags, uint32_t* U,
                  int32_t* cnt, int64_t* seg_off, int64_t* seg_total, int64_t* volume, char* ws, const WsLayout& L,
                  cudaStream_t st);
int launch_demand_pack(const sparsp_shape& s, const Geometry& g, const uint32_t* mask, const int32_t* rank, int P,
                       int flags, const void* K, const void* V, uint32_t* U, int32_t* cnt, int64_t* seg_off,
                       int64_t* seg_total, int64_t* volume, void* packed, int64_t capacity, const int64_t* dst_base,
                       char* ws, const WsLayout& L, cudaStream_t st);
int launch_pack_segment(const sparsp_shape& s, const Geometry& g, const uint32_t* U, const int32_t* rank, int P,
                        int consumer, int producer, const int64_t* seg_off, const int32_t* cnt, const void* K,
                        const void* V, void* dst, int64_t capacity, char* ws, const WsLayout& L, cudaStream_t st);
int launch_attn(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, const void* V,
                const uint32_t* mask, float scale, void* O, float* lse, char* ws, const WsLayout& L,
                cudaStream_t st);

int launch_attn_packed(const sparsp_shape& s, const Geometry& g, const void* Q, const void* K, const void* V,
                       const uint32_t* mask, const int32_t* rank, int P, int consumer, const uint32_t* U,
                       const int64_t* seg_off, const int64_t* seg_total, const void* packed, int64_t capacity,
                       const int64_t* dst_base, float scale, void* O, float* lse, char* ws, const WsLayout& L,
                       cudaStream_t st);
int launch_hop_mask(const Geometry& g, const uint32_t* mask, const int32_t* rank, int consumer, int producer,
                    int head_begin, int head_end, uint32_t* hop, cudaStream_t st);
int launch_wait_timeout(char* ws, const WsLayout& L, long long limit_cycles, cudaStream_t st);
int launch_attn_merge(const sparsp_shape& s, const Geometry& g, const void* Oa, const float* la, const void* Ob,
                      const float* lb, void* O, float* lse, const int32_t* rank, int consumer, int head_begin,
                      int head_end, cudaStream_t st);

}  // namespace sparsp
