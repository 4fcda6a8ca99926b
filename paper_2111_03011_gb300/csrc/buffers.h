// Rules on the memory that callers hand in: which buffers a kernel may use
// where they lie.  Host-only, no CUDA headers.
#pragma once

#include <cstddef>
#include <cstdint>

namespace tn {

// Whether [a, a + na) and [b, b + nb) share a byte.
inline bool ranges_overlap(const void* a, size_t na, const void* b, size_t nb) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return na > 0 && nb > 0 && x < y + nb && y < x + na;
}

// Whether a kernel that moves `align` bytes at a time may use the buffer at p.
// A caller's element type can need less: C's double _Complex, std::complex<double>
// and NumPy's complex128 start on 8 bytes, a kernel's 16-byte store does not.
inline bool kernel_aligned(const void* p, size_t align) { return (uintptr_t)p % align == 0; }

}  // namespace tn
