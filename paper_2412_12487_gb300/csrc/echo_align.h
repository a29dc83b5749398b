// echo_align.h -- whether kernels may read a caller's host arrays where they lie.  A copy
// takes any address, a device load only multiples of its element's size (anything else ends
// the CUDA context), and callers may pass arrays at any byte (a view into a mapped file, a
// packed record).  No CUDA dependency, so the test is compiled for the host and checked there.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <initializer_list>

namespace echo {

// every one of `arrays` starts on a multiple of `size`, its elements' size
inline bool elements_aligned(size_t size, std::initializer_list<const void *> arrays) {
  for (const void *p : arrays)
    if (reinterpret_cast<uintptr_t>(p) % size != 0) return false;
  return true;
}

}  // namespace echo
