// alloc.h -- buffers from a caller's allocator, of whatever alignment.
#pragma once
#include <cstddef>
#include <cstdint>

#include "../../include/dsdna.h"

namespace dsdna {

// `bytes` on a 16-byte boundary (kernels load and store 16 bytes at a time) from
// the caller's allocator; *raw is what to release.  A block that starts elsewhere
// is returned and one with room to align asked for.  Null when out of memory.
inline void* alloc16(const dsdna_allocator& al, size_t bytes, void** raw) {
  *raw = al.alloc(bytes, al.user);
  if (*raw && (uintptr_t)*raw % 16 != 0) {
    al.release(*raw, al.user);
    *raw = al.alloc(bytes + 15, al.user);
  }
  return (void*)(((uintptr_t)*raw + 15) & ~(uintptr_t)15);
}

}  // namespace dsdna
