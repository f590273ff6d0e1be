// Clusters of thread blocks: barriers, and the shared memory of the other blocks.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace wersa {

constexpr int kMaxCluster = 16;   // blocks of a cluster (more than 8 are opt-in)

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// The two halves of a barrier of all threads of the cluster's blocks: what was written to shared memory before is visible behind.
__device__ __forceinline__ void cluster_release() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_acquire() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// The same, nothing released: the blocks of the cluster have begun (their shared memory may be written to).
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t shared_addr(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }
// The same place in the shared memory of block `rank`.  (Blocks only write to one another and read their own memory, and what is
// more than a few hundred bytes goes as bulk copies.  The sums over S' of 3 x 130, m = 256 by reads of the peers' memory, 16 bytes a
// lane, a row's side by side: 17 us a forward, row by row 26; by copies 13.  By 8-byte stores from the accumulators 14.)
__device__ __forceinline__ uint32_t peer_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void peer_store2(uint32_t addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// `bytes` (a multiple of 16, not 0) of this block's shared memory to another block's, reported to a barrier over there.  What was
// written here has to be fenced for the copy engine; the block may not end before the copy has (a barrier of the cluster).
__device__ __forceinline__ void peer_copy(uint32_t dst, uint32_t src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "r"(src), "r"(bytes),
               "r"(bar) : "memory");
}

// Once per CUDA context, ahead of the first launch (a wersa_ctx is created): 0.4 us a call, of which a forward that waits for the host has none
// to spare (1 x 2531, m = 128 16.7 us with a plain launch, 17.4 with two of these at each launch of the mean pool).
template <typename K> inline cudaError_t prepare_cluster(K kernel, size_t smem, int blocks) {
  const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return err != cudaSuccess || blocks <= 8 ? err : cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}
// How many clusters of `blocks` the device holds at once (0: none, or no device).
template <typename K> inline int clusters_at_once(K kernel, int threads, size_t smem, int blocks) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = blocks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (prepare_cluster(kernel, smem, blocks) == cudaSuccess && cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess)
    return clusters;
  cudaGetLastError();   // a failed query leaves no sticky error behind
  return 0;
}
// The current CUDA context's number, which no other context of the process ever has; 0: none, or not to be had.
inline unsigned long long current_context_id() {
  using Fn = CUresult (*)(CUcontext, unsigned long long*);
  static const Fn fn = []() -> Fn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuCtxGetId", &p, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<Fn>(p);
    cudaGetLastError();
    return nullptr;
  }();
  unsigned long long id = 0;
  return fn != nullptr && fn(nullptr, &id) == CUDA_SUCCESS ? id : 0;
}
// What clusters_at_once answered, for the CUDA context that it was asked in: the answer and the kernel's attributes belong to that,
// not to the device, and another context (one more of the driver API's, the next one after a reset) asks again.  wersa_create
// takes 30 to 140 us where it asks, 1.5 where it does not.  An answer of none is not kept: the query may have failed for a reason that
// passes.
struct KnownClusters {
  std::atomic<unsigned long long> word{0};   // context number << 16 | answer
  template <typename Ask> int get(Ask&& ask) {
    const unsigned long long id = current_context_id(), w = word.load(std::memory_order_acquire);
    if (id != 0 && w >> 16 == id) return (int)(w & 0xFFFF);
    const int clusters = ask();
    if (id != 0 && id >> 48 == 0 && clusters > 0 && clusters <= 0xFFFF)
      word.store(id << 16 | (unsigned long long)clusters, std::memory_order_release);
    return clusters;
  }
};
// A launch like launch_after's whose grid's first dimension is one cluster.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = grid.x;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

}  // namespace wersa
