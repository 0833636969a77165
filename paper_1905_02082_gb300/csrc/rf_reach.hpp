// Which of a caller's buffers the kernels may use directly (host code; the
// attributes come from `attributes`, cudaPointerGetAttributes or a test's).
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

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

// Images are copied 16 bytes at a time; byte by byte a kernel is slower than
// the copy engine (an unaligned page-locked frame of 640x480: 23 us against
// 13).  Poses and infos are accessed in 8 bytes, which a kernel may do only at
// such an address.
constexpr size_t kImageAlign = 16, kWordAlign = 8;

// Whether the staging kernels take the buffer: reachable, at a multiple of `align`.
template <class Attributes>
bool staged_by_kernel(const void* p, size_t bytes, size_t align, int device, Attributes&& attributes) {
  return reinterpret_cast<uintptr_t>(p) % align == 0 && reachable(p, bytes, device, attributes);
}

}  // namespace rf
