// The fused step's kernels for double storage and 64 threads per CTA (fused.cuh), a
// translation unit of their own so that they compile beside the others.
#include "fused.cuh"

namespace ifd {

void launch_fused_double_64(const FusedArgs &a, int grid, cudaStream_t s) {
  launch_fused_nt<double, 64>(a, grid, s);
}
int blocks_per_sm_double_64() { return blocks_per_sm_nt<double, 64>(); }
int smem_double_64() { return fused_smem_size<double, 64>(); }

}  // namespace ifd
