// Copies of a handle's planes to and from the caller's buffer (checkpoints, kept
// intermediates): which of them a kernel makes, and which the copy engine.
#pragma once
#include <cstdint>

namespace ifd {

// Copies of up to three segments of memory.
struct CopyArgs {
  const void *src[3];
  void *dst[3];
  int64_t bytes[3];
};

// One kernel (k_copy) takes all segments while they are small, where the launches
// of three copies cost more than the bytes: the state of a 257^2 cavity 2.9 us
// against 16.5. Above this size in all they do not count.
constexpr int64_t COPY_MOST = int64_t(64) << 20;

// `here`: the caller's buffer is memory of the handle's own device. Any other
// (another device, which a kernel reaches only with peer access; the host) is left
// to the copy engine whatever its size, and so are segments that are not on
// 16-byte boundaries or not whole doubles.
inline bool copy_by_kernel(const CopyArgs &a, bool here) {
  int64_t total = 0;
  bool plain = here;
  for (int k = 0; k < 3; ++k) {
    total += a.bytes[k];
    plain = plain && ((uintptr_t(a.src[k]) | uintptr_t(a.dst[k])) & 15) == 0 && a.bytes[k] % 8 == 0;
  }
  return plain && total <= COPY_MOST;
}

}  // namespace ifd
