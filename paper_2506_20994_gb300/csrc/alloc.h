// Device buffers that a handle allocates together.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <initializer_list>

#include "../../include/axhelm.h"

namespace ax {

struct Buffer {
  void **p;
  size_t bytes;
  template <typename T>
  Buffer(T **ptr, size_t count) : p(reinterpret_cast<void **>(ptr)), bytes(count * sizeof(T)) {}
  Buffer(void **ptr, size_t size) : p(ptr), bytes(size) {}
};

inline void free_all(std::initializer_list<Buffer> group) {
  for (const Buffer &b : group) {
    cudaFree(*b.p);
    *b.p = nullptr;
  }
}

// Every buffer of the group anew, or none of them: what they held before is
// freed first, and after a failure every pointer is null, so that a handle
// never keeps a half-made group or a pointer to freed memory.
inline int alloc_all(std::initializer_list<Buffer> group) {
  free_all(group);
  for (const Buffer &b : group) {
    if (cudaMalloc(b.p, std::max<size_t>(b.bytes, 1)) != cudaSuccess) {
      (void)cudaGetLastError();
      *b.p = nullptr;
      free_all(group);
      return AX_ENOMEM;
    }
  }
  return AX_OK;
}

}  // namespace ax
