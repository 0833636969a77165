// Which of a caller's buffers the kernels may use directly (host code; the
// attributes come from `attributes`, cudaPointerGetAttributes or a test's).
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>

namespace rf {

// Whether kernels on `device` may read and write the `bytes` bytes at p: its
// own memory, managed memory, and page-locked host memory that is mapped at
// its own address, from the first byte to the last (a host range may be
// registered in part).  Memory of another device is left to the copy engine,
// which needs no peer access, and so is everything unknown, which a copy
// refuses with an error where a kernel would fault.
template <class Attributes>
bool reachable(const void* p, size_t bytes, int device, Attributes&& attributes) {
  cudaPointerAttributes at;
  if (attributes(&at, p) != cudaSuccess) return false;
  switch (at.type) {
    case cudaMemoryTypeDevice: return at.device == device;
    case cudaMemoryTypeManaged: return true;
    case cudaMemoryTypeHost: {
      const void* last = static_cast<const char*>(p) + (bytes > 0 ? bytes - 1 : 0);
      cudaPointerAttributes end;
      return at.devicePointer == p && attributes(&end, last) == cudaSuccess && end.type == cudaMemoryTypeHost &&
             end.devicePointer == last;
    }
    default: return false;
  }
}

}  // namespace rf
