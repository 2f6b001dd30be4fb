// Dispatch of the fused step over its storage types and CTA widths (fused.cuh).
#include "internal.h"

namespace ifd {

#define IFD_FUSED(T, NT)                                                  \
  void launch_fused_##T##_##NT(const FusedArgs &a, int grid, cudaStream_t s); \
  int blocks_per_sm_##T##_##NT();                                         \
  int smem_##T##_##NT();
IFD_FUSED(float, 64)
IFD_FUSED(float, 128)
IFD_FUSED(float, 256)
IFD_FUSED(double, 64)
IFD_FUSED(double, 128)
IFD_FUSED(double, 256)
#undef IFD_FUSED

#define IFD_FUSED(T)                                                              \
  template <> bool launch_fused<T>(const FusedArgs &a, int nt, int grid, cudaStream_t s) { \
    switch (nt) {                                                                 \
      case 64: launch_fused_##T##_64(a, grid, s); return true;                    \
      case 128: launch_fused_##T##_128(a, grid, s); return true;                  \
      case 256: launch_fused_##T##_256(a, grid, s); return true;                  \
    }                                                                             \
    return false;                                                                 \
  }                                                                               \
  template <> int fused_blocks_per_sm<T>(int nt) {                                \
    return nt == 64 ? blocks_per_sm_##T##_64()                                    \
                    : (nt == 128 ? blocks_per_sm_##T##_128()                      \
                                 : (nt == 256 ? blocks_per_sm_##T##_256() : 0));  \
  }                                                                               \
  template <> int fused_smem_bytes<T>(int nt) {                                   \
    return nt == 64 ? smem_##T##_64()                                             \
                    : (nt == 128 ? smem_##T##_128() : (nt == 256 ? smem_##T##_256() : -1)); \
  }
IFD_FUSED(float)
IFD_FUSED(double)
#undef IFD_FUSED

}  // namespace ifd
