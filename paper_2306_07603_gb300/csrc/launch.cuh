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
#include <cuda_runtime.h>

namespace ifd {

__device__ __forceinline__ void previous_done() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
__device__ __forceinline__ void dependents_may_start() {
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

template <class Args>
inline void launch_after(void (*kernel)(Args), int grid, int block, int smem, cudaStream_t s,
                         const Args &args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(block));
  cfg.dynamicSmemBytes = size_t(smem);
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, args);
}

}  // namespace ifd
