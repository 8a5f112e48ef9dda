// Device memory of the library's objects and the identity of contexts (host declarations only).
#pragma once

#include <stddef.h>

#include <cuda_runtime.h>

namespace lbmhd_gpu {

// Device memory of handles (lbmhd_memory.cu).  device_free keeps a block for later device_alloc calls
// of the same size if `idle`, i.e. if no work on it can be in flight any more.
cudaError_t device_alloc(void** out, size_t bytes);
void device_free(void* ptr, bool idle);

// cudaMalloc and cudaMallocAsync that give back the kept blocks of the device and try again when there
// is no memory left: every other allocation of the library goes through these.  Free with cudaFree and
// cudaFreeAsync.
cudaError_t device_malloc(void** out, size_t bytes);
cudaError_t device_malloc_async(void** out, size_t bytes, cudaStream_t s);
template <typename T>
cudaError_t device_malloc(T** out, size_t bytes) {
  return device_malloc(reinterpret_cast<void**>(out), bytes);
}

// Driver function `name` (as of driver API `version`), reached through the runtime's entry point --
// the library does not link libcuda -- or nullptr (lbmhd_noalloc.cu).
void* driver_entry(const char* name, int version);

// Identifier of the calling thread's current context, unique for the life of the process; false if
// it cannot be had (lbmhd_noalloc.cu).
bool current_context_id(unsigned long long* id);

}  // namespace lbmhd_gpu
