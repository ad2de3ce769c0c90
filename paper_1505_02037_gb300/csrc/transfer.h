// Which host arrays a kernel may read or write where a copy call would do.
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace lbnr {

// Whether the `bytes` at p, whole doubles, lie in the one page-locked range
// [start, start + size) and on addresses that 8-byte loads and stores can take.
// Both ends in page-locked memory are not enough: they can belong to two
// registrations with pageable memory between them, and a kernel that touches
// that faults where a copy call returns an error.
inline bool kernel_reaches(uintptr_t p, size_t bytes, uintptr_t start, size_t size) {
  return bytes > 0 && p % 8 == 0 && bytes % 8 == 0 && p >= start && bytes <= size &&
         p - start <= size - bytes;
}

}  // namespace lbnr
