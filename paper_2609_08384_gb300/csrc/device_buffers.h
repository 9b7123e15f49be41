// Which buffers of a caller a kernel may copy fields from and to.
#pragma once

#include <stdint.h>

#include <cuda_runtime.h>

namespace brahms {

// Whether a kernel of the current device can read (or write) n buffers of
// `bytes` bytes as 16-byte pairs: device memory of this device, aligned, apart
// from the library's memory [lo, hi) and, when written, from each other.
// Otherwise the driver's copies move the fields one after another.
inline bool kernel_can_copy(const void* const* ptrs, int n, size_t bytes, const void* lo, const void* hi, bool written) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  for (int f = 0; f < n; ++f) {
    const uintptr_t p = (uintptr_t)ptrs[f];
    if ((p & 15) != 0 || (p < (uintptr_t)hi && (uintptr_t)lo < p + bytes)) return false;
    for (int g = 0; written && g < f; ++g) {
      const uintptr_t q = (uintptr_t)ptrs[g];
      if (p < q + bytes && q < p + bytes) return false;
    }
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, ptrs[f]) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    if (at.type != cudaMemoryTypeDevice || at.device != dev) return false;
  }
  return true;
}

}  // namespace brahms
