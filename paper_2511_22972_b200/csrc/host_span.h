// Which host buffers the kernels may read where they lie.  Host arithmetic only.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace fly {

// What the driver knows about the pointer to a buffer (all zero: nothing, as about pageable memory).
struct HostSpan {
  unsigned type;        // CUmemorytype: 1 = host
  uint64_t device;      // the address under which kernels see the pointer
  uint64_t start;       // of the one allocation or registration that the pointer lies in ...
  size_t size;          // ... and its bytes
  unsigned managed;     // moves between host and device: copied
};

// A kernel that leaves the mapping faults, where a copy is refused: the whole buffer has to lie in one page-locked range, and
// not its first byte alone.  Nor can a kernel load elements off their own alignment, which a copy moves to an aligned place.
inline bool readable_in_place(const HostSpan& s, const void* host, size_t bytes, size_t element) {
  const uint64_t p = (uint64_t)(uintptr_t)host;
  return p % element == 0 && s.type == 1 && !s.managed && s.device == p && s.start <= p && bytes <= s.size && p - s.start <= s.size - bytes;
}

}  // namespace fly
