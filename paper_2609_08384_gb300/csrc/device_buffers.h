// Which buffers of a caller a kernel may copy fields from and to.
#pragma once

#include <stddef.h>
#include <stdint.h>

#include <cuda.h>
#include <cuda_runtime.h>

namespace brahms {

// Where the bytes [p, p + bytes) lie: in the allocation that holds p, in
// allocations that follow one another without a gap, or beyond memory that is
// there.  allocation_of(address, &base, &size) finds an address's allocation,
// false if it has none.
enum class Extent { kWhole, kPieces, kShort, kUnknown };
template <class AllocationOf>
Extent extent_of(uintptr_t p, size_t bytes, AllocationOf allocation_of) {
  uintptr_t base = 0;
  size_t size = 0;
  if (!allocation_of(p, &base, &size) || p < base || p - base >= size) return Extent::kUnknown;
  uintptr_t at = base + size;  // first address behind the memory known to be there
  if (bytes <= at - p) return Extent::kWhole;
  if (p + bytes < p) return Extent::kShort;
  while (at < p + bytes) {
    if (!allocation_of(at, &base, &size) || at < base || at - base >= size) return Extent::kShort;
    at = base + size;
  }
  return Extent::kPieces;
}

// A function of the driver's, NULL if it has none of that name.
template <class F>
F driver_function(const char* name) {
  void* f = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion(name, &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess) {
    cudaGetLastError();
    f = nullptr;
  }
  return reinterpret_cast<F>(f);
}

// The device allocation that holds an address, or the piece of memory mapped there.
inline bool device_allocation_of(uintptr_t p, uintptr_t* base, size_t* size) {
  typedef CUresult (*Fn)(CUdeviceptr*, size_t*, CUdeviceptr);
  static const Fn range = driver_function<Fn>("cuMemGetAddressRange");
  CUdeviceptr b = 0;
  if (!range || range(&b, size, (CUdeviceptr)p) != CUDA_SUCCESS) return false;
  *base = (uintptr_t)b;
  return true;
}

// Whether [p, p + bytes) lies in one range of addresses: an allocation, or a range
// reserved for pieces mapped one after another.
inline bool one_address_range(uintptr_t p, size_t bytes) {
  typedef CUresult (*Fn)(void*, CUpointer_attribute, CUdeviceptr);
  static const Fn attribute = driver_function<Fn>("cuPointerGetAttribute");
  CUdeviceptr start = 0;
  size_t size = 0;
  return attribute && attribute(&start, CU_POINTER_ATTRIBUTE_RANGE_START_ADDR, (CUdeviceptr)p) == CUDA_SUCCESS &&
         attribute(&size, CU_POINTER_ATTRIBUTE_RANGE_SIZE, (CUdeviceptr)p) == CUDA_SUCCESS && p >= start &&
         p - start <= size && bytes <= size - (p - start);
}

// How n buffers of `bytes` bytes that a caller calls device buffers are read (or
// written): by a kernel as 16-byte pairs where they are device memory of the
// current device, each inside one allocation, aligned, apart from the library's
// memory [lo, hi) and, when written, from each other; otherwise by the driver's
// copies, one after another.  A buffer that ends before its last byte, or runs on
// into another allocation, is refused, as the driver's copies refuse it: a kernel
// would read or write past its end.
enum class Route { kKernel, kDriver, kRefuse };
inline Route device_route(const void* const* ptrs, int n, size_t bytes, const void* lo, const void* hi, bool written) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return Route::kDriver;
  Route route = Route::kKernel;
  for (int f = 0; f < n; ++f) {
    const uintptr_t p = (uintptr_t)ptrs[f];
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, ptrs[f]) != cudaSuccess) {
      cudaGetLastError();
      route = Route::kDriver;
      continue;
    }
    const Extent e = at.type == cudaMemoryTypeDevice ? extent_of(p, bytes, device_allocation_of) : Extent::kUnknown;
    if (e == Extent::kShort || (e == Extent::kPieces && !one_address_range(p, bytes))) return Route::kRefuse;
    if (e != Extent::kWhole || at.device != dev || (p & 15) != 0 || (p < (uintptr_t)hi && (uintptr_t)lo < p + bytes))
      route = Route::kDriver;
    for (int g = 0; written && g < f; ++g) {
      const uintptr_t q = (uintptr_t)ptrs[g];
      if (p < q + bytes && q < p + bytes) route = Route::kDriver;
    }
  }
  return route;
}

}  // namespace brahms
