// common.cuh -- device helpers shared by the library's kernels (sm_103a).
#pragma once
#include <limits.h>

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "dreams.h"

namespace dreams {

// Thread-local record of the last failing CUDA call (dreams_last_cuda_error).
void set_last_cuda_error(cudaError_t e);

// Streaming multiprocessors of the current device (cached per device).
int num_sms();

// Raises a kernel's maximum dynamic shared memory on the current device to at
// least `bytes` (the attribute is set again only for a larger request); safe
// to call from several host threads.
dreams_status_t ensure_max_dynamic_smem(const void *func, int bytes);

// The stall test hook (dreams_test_set_stall) as it applies to one kernel
// family: the index of the first withheld copy (-1: none) and the limit of
// every pipeline wait (2 s unless the hook shortens it).
void test_stall(int32_t kernel, int32_t *stall_at, uint64_t *wait_ns);

inline dreams_status_t check_launch() {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_last_cuda_error(e);
    return DREAMS_ERR_CUDA;
  }
  return DREAMS_OK;
}

// Every kernel of the library is launched as a programmatic dependent of the
// launch before it on the stream: its CTAs may become resident while that grid
// drains, and each begins with grid_wait(), which returns once that grid has
// completed and its writes are visible. A kernel whose successor is the next
// stage of the same call lets it start early (launch_successor, after the wait,
// so that at most one grid ahead of a running CTA is unfinished): the merge of
// the attention's partials launched so takes 1.2 us off 18.7. The last kernel
// of a call leaves its successor to its CTAs' exits: what comes next may stream
// with a chip's worth of CTAs, which would fill the SMs that are free first and
// leave the others idle (batched attention, then the verification: 131.0
// against 110.3 us; a 3392-slot attention and a batched verification 74.8
// against 57.0).
// The sampling statistics let the selection start at the end of their work
// (earlier, or only with the exits, 240 rows of 32003 f32 took 18 against 15
// us); the importance sums leave it to the exits (103.3 against 105.3 us).
// A kernel that reads global memory before its wait may read only what its own
// predecessor's inputs were (the walk's tree arrays), and reads it through L2
// (__ldcg): L1 may hold older lines until the wait.
// cluster: the CTAs of a cluster; 0 for a kernel without clusters. (A cluster of
// one CTA needs the attribute too: without it the walk's st.async faulted as an
// illegal instruction.)
template <typename... Params, typename... Args>
dreams_status_t launch_clusters(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                int cluster, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = unsigned(cluster);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 0 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
  if (e != cudaSuccess) {
    set_last_cuda_error(e);
    return DREAMS_ERR_CUDA;
  }
  return check_launch();
}

template <typename... Params, typename... Args>
dreams_status_t launch_kernel(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args... args) {
  return launch_clusters(kernel, grid, block, smem, stream, 0, args...);
}

// Waits until the preceding grid has completed and its writes are visible.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next launch on the stream start once every CTA has come here.
__device__ __forceinline__ void launch_successor() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Every thread of every CTA of the cluster: release this CTA's shared-memory
// writes (local and remote), then wait for all CTAs (a superset of
// __syncthreads).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}

__device__ __forceinline__ uint32_t cluster_addr(const void *local_ptr, uint32_t rank) {
  const uint32_t a = static_cast<uint32_t>(__cvta_generic_to_shared(local_ptr));
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  return ra;
}

// A read-only global load issued where it stands (the compiler may not sink it
// to the value's first use), so that its latency overlaps the work in between.
__device__ __forceinline__ int ld_issue_now(const int32_t *ptr) {
  int v;
  asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(ptr));
  return v;
}

inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

__device__ __forceinline__ void flag(int32_t *status_word, int32_t bits) {
  if (status_word != nullptr) atomicOr(status_word, bits);
}

// ---------------------------------------------------------------- tree checks
// A tree row is valid when 1 <= T <= T_max, parent[0] == -1 and
// 0 <= parent[i] < i for 0 < i < T.

// ---------------------------------------------------------------- PTX wrappers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Order-preserving integer key of an f32 bit pattern for the argmax order:
// greater value -> greater key, +0 == -0, NaN above every number.
__device__ __forceinline__ int order_key(uint32_t u) {
  const uint32_t mag = u & 0x7fffffffu;
  if (mag > 0x7f800000u) return INT_MAX;  // NaN
  if (mag == 0u) return 0;                // +0 and -0
  const int s = static_cast<int>(u);
  return s ^ ((s >> 31) & 0x7fffffff);
}

// (key, index) packed so that a 64-bit max keeps the greater key, then the
// lower index.
__device__ __forceinline__ unsigned long long pack_key_idx(int key, int idx) {
  return (static_cast<unsigned long long>(static_cast<uint32_t>(key) ^ 0x80000000u) << 32) |
         static_cast<unsigned long long>(~static_cast<uint32_t>(idx));
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t *>(&v);
}

}  // namespace dreams
