// Where a caller's array lies (host arithmetic on addresses, no CUDA).
#pragma once

#include <stddef.h>
#include <stdint.h>

namespace pic {

// n elements of `size` bytes from p lie inside the allocation of `bytes` bytes from base.
inline bool array_inside(uintptr_t base, size_t bytes, uintptr_t p, int64_t n, size_t size) {
  return n >= 0 && p >= base && p - base <= bytes && (uint64_t)n <= (bytes - (p - base)) / size;
}

// n elements of `size` bytes from p (no wrap: they lie in an allocation) share no byte with the
// `bytes` bytes from q.
inline bool array_apart(uintptr_t p, int64_t n, size_t size, uintptr_t q, size_t bytes) {
  const size_t len = (size_t)n * size;
  return len == 0 || bytes == 0 || (p < q ? q - p >= len : p - q >= bytes);
}

}  // namespace pic
