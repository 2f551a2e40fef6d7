// Read-out into the caller's memory.
//
// A fresh numpy (or malloc) array of a few MB has no pages yet.  Left to the
// device copy, each missing page is a fault that the GPU raises and waits for:
// 65 MB of positions and velocities into six new arrays took 53 ms, 50 us per
// 64 KB page, where the same copy into present pages takes 0.8 ms.  So the
// host makes the pages present first: 23 ms for pages the machine has never
// given out, 2 ms for recycled ones, whether by one thread or by sixteen.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>
#include <unistd.h>

namespace vcsgc {

// smallest read-out whose pages are looked at: heap memory in use serves
// smaller ones
constexpr size_t READOUT_MIN_BYTES = 32 << 10;

// Makes the pages of n buffers of `bytes` each present without changing their
// contents (null: none).  Only for memory that CUDA does not know: pinned and
// managed memory is left alone, a device pointer is left for the copy to refuse.
template <typename T>
inline void make_present(T* const* p, int n, size_t bytes) {
  if (bytes < READOUT_MIN_BYTES) return;
  const size_t page = (size_t)sysconf(_SC_PAGESIZE);
  char* buf[8];
  int nb = 0;
  for (int q = 0; q < n && nb < 8; ++q) {
    if (!p[q]) continue;
    cudaPointerAttributes at;
    if (cudaPointerGetAttributes(&at, p[q]) != cudaSuccess) cudaGetLastError();
    else if (at.type == cudaMemoryTypeUnregistered) buf[nb++] = reinterpret_cast<char*>(p[q]);
  }
  for (int q = 0; q < nb; ++q) {
    for (size_t o = 0; o < bytes; o += page) __atomic_fetch_or(buf[q] + o, 0, __ATOMIC_RELAXED);
    __atomic_fetch_or(buf[q] + bytes - 1, 0, __ATOMIC_RELAXED);
  }
}

// device -> caller's host memory, on the stream
inline cudaError_t read_back(void* dst, const void* src, size_t bytes, cudaStream_t st) {
  make_present(&dst, 1, bytes);
  return cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToHost, st);
}

}  // namespace vcsgc
