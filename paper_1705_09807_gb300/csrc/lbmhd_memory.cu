// Device memory of handles, with the blocks of freed handles kept for the next ones.
//
// A program that makes many short runs creates and frees a handle per run, and cudaMalloc and
// cudaFree (which map and unmap the memory and wait for the whole device) then take a large part of
// it: 0.81 ms for the two population copies of a 2048^2 binary32 grid and 0.06 ms for each small
// block, against 2.8 ms for twenty steps.  Taking both copies and the small blocks from freed ones
// shortened that job (page-locked fields in, twenty steps, snapshot to the host) from 5.54 to 4.53 ms.
//
// Rules.  A block enters the cache only when no work on it can be in flight (the caller has
// synchronised the stream that used it) and only in the context it was allocated in, so it can be
// handed to any stream.  The cache holds at most kMaxCached bytes (the oldest blocks go first), is
// emptied when an allocation fails, and by lbmhd_release_cached_memory.  Blocks are matched by exact
// size; their contents are not cleared (nor are cudaMalloc's).  A context that was destroyed
// (cudaDeviceReset) took its blocks with it: they are forgotten, never freed.  All state is behind
// one mutex.
#include <cuda_runtime.h>

#include <list>
#include <mutex>
#include <new>
#include <unordered_map>

#include "lbmhd.h"
#include "lbmhd_internal.cuh"

namespace lbmhd_gpu {
namespace {

constexpr size_t kMaxCached = (size_t)1 << 30;

struct Block {
  void* ptr;
  size_t bytes;
  int device;
  unsigned long long context;
};

std::mutex g_mutex;
std::list<Block> g_cached;                   // oldest first
std::unordered_map<void*, Block> g_in_use;   // blocks that may be cached when they are freed
size_t g_cached_bytes = 0;

// Identity of the current device and context; false if it cannot be had (nothing is cached then).
bool here(int* device, unsigned long long* context) {
  return cudaGetDevice(device) == cudaSuccess && current_context_id(context);
}

// Take blocks out of the cache until at most `most` bytes of it are left.
void shrink(size_t most) {
  int device = 0;
  unsigned long long context = 0;
  const bool known = here(&device, &context);
  for (auto it = g_cached.begin(); it != g_cached.end() && g_cached_bytes > most;) {
    // another device's block cannot be checked against its context from here: left for its own turn
    if (known && it->device != device) {
      ++it;
      continue;
    }
    if (known && it->context == context) cudaFree(it->ptr);
    g_cached_bytes -= it->bytes;
    it = g_cached.erase(it);
  }
}

}  // namespace

cudaError_t device_alloc(void** out, size_t bytes) {
  *out = nullptr;
  std::lock_guard<std::mutex> lock(g_mutex);
  int device = 0;
  unsigned long long context = 0;
  const bool known = here(&device, &context);
  try {
    if (known) {
      for (auto it = g_cached.begin(); it != g_cached.end(); ++it) {
        if (it->bytes != bytes || it->device != device || it->context != context) continue;
        g_in_use.emplace(it->ptr, *it);
        *out = it->ptr;
        g_cached_bytes -= it->bytes;
        g_cached.erase(it);
        return cudaSuccess;
      }
    }
    cudaError_t e = cudaMalloc(out, bytes);
    if (e == cudaErrorMemoryAllocation && g_cached_bytes > 0) {
      cudaGetLastError();
      shrink(0);
      e = cudaMalloc(out, bytes);
    }
    if (e != cudaSuccess) {
      *out = nullptr;
      return e;
    }
    // (the first allocation of a process makes its context)
    if (known || here(&device, &context)) g_in_use[*out] = Block{*out, bytes, device, context};
    return cudaSuccess;
  } catch (const std::bad_alloc&) {  // host memory for the bookkeeping
    if (*out) return cudaSuccess;    // the block is good, it will not be cached
    return cudaErrorMemoryAllocation;
  }
}

void device_free(void* ptr, bool idle) {
  if (!ptr) return;
  std::lock_guard<std::mutex> lock(g_mutex);
  int device = 0;
  unsigned long long context = 0;
  auto it = g_in_use.find(ptr);
  if (it != g_in_use.end()) {
    const Block b = it->second;
    g_in_use.erase(it);
    if (idle && b.bytes <= kMaxCached && here(&device, &context) && b.device == device && b.context == context) {
      try {
        g_cached.push_back(b);
        g_cached_bytes += b.bytes;
        shrink(kMaxCached);
        return;
      } catch (const std::bad_alloc&) {
      }
    }
  }
  cudaFree(ptr);
}

}  // namespace lbmhd_gpu

extern "C" void lbmhd_release_cached_memory(void) {
  std::lock_guard<std::mutex> lock(lbmhd_gpu::g_mutex);
  lbmhd_gpu::shrink(0);
}
