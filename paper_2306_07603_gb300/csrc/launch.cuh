// Kernel launches whose start overlaps the end of the kernel before them in the
// stream (programmatic dependent launch).
//
// A step is one to three short kernels that each read what the one before
// wrote. Launched plainly, each pays the drain of its predecessor, the launch
// latency and its own start-up in turn. Launched with launch_after, a
// kernel's blocks may become resident once every block of its predecessor
// has called dependents_may_start() or ended, and run up to previous_done(),
// which returns when the predecessor has completed and its writes are visible.
// Rules for such kernels: every thread calls previous_done() before its
// first access to memory that any kernel or copy of the stream writes (tables
// uploaded at creation are not), and none returns before it.
#pragma once
#include <cooperative_groups.h>
#include <cuda_runtime.h>

namespace ifd {

__device__ __forceinline__ void previous_done() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
__device__ __forceinline__ void dependents_may_start() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// Shared memory of the first block of a cluster of CS blocks. A block's shared
// memory may be accessed from another one only once that block is known to run
// (being launched together does not say so), and until it ends. So every thread
// calls cluster_arrive() at the start of the kernel and cluster_running(), which
// returns when all of the cluster's threads have done so, before the first use of
// cluster_at(): the address of p, in this block's shared memory, in that of the
// first block. The arrival orders no memory; what lies between the two hides it.
// cluster_done() is the barrier after which the first block reads what the others
// wrote there. Every thread of the block calls each of them, or none does.
template <int CS>
__device__ __forceinline__ void cluster_arrive() {
  if constexpr (CS > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::);
}
template <int CS>
__device__ __forceinline__ void cluster_running() {
  if constexpr (CS > 1) asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");
}
template <int CS>
__device__ __forceinline__ double *cluster_at(double *p) {
  if constexpr (CS == 1)
    return p;
  else
    return cooperative_groups::this_cluster().map_shared_rank(p, 0);
}
template <int CS>
__device__ __forceinline__ void cluster_done() {
  if constexpr (CS == 1)
    __syncthreads();
  else
    cooperative_groups::this_cluster().sync();
}

template <class Args>
inline void launch_after(void (*kernel)(Args), int grid, dim3 block, int smem, cudaStream_t s,
                         const Args &args, int cluster = 1) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = size_t(smem);
  cfg.stream = s;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim = {unsigned(cluster), 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  cudaLaunchKernelEx(&cfg, kernel, args);
}

}  // namespace ifd
