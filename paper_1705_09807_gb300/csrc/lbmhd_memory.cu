// Device memory of handles, with the blocks of freed handles kept for the next ones.
//
// A program that makes many short runs creates and frees a handle per run, and cudaMalloc and
// cudaFree (which map and unmap the memory and wait for the whole device) then take a large part of
// it: 0.81 ms for the two population copies of a 2048^2 binary32 grid and 0.06 ms for each small
// block, against 2.8 ms for twenty steps.  Taking both copies and the small blocks from freed ones
// shortened that job (page-locked fields in, twenty steps, snapshot to the host) from 5.54 to 4.53 ms.
//
// Rules.  A block enters the cache only when no work on it can be in flight (the caller has
// synchronised the stream that used it), only in the context it was allocated in, so it can be
// handed to any stream, and only if that is its device's primary context (the runtime's own).  The
// cache holds at most kMaxCached bytes (the oldest blocks go first), gives a device's blocks back when
// an allocation of the library there finds no memory, and all blocks by lbmhd_release_cached_memory.  Blocks are matched by
// exact size; their contents are not cleared (nor are cudaMalloc's).  A block is freed in its own
// context, whatever the calling thread has current -- another device, another context, or none
// yet -- and its record is dropped without that only if its context is known to be gone: a
// device has one primary context at a time, so when it has none, or one with another identifier, the
// block went with the former one (cudaDeviceReset).  All state is behind one mutex.
#include <cuda.h>
#include <cuda_runtime.h>

#include <list>
#include <mutex>
#include <new>
#include <unordered_map>

#include "lbmhd.h"
#include "lbmhd_memory.h"

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

// Identity of the calling thread's device and context; a thread that has no context yet (one that
// has made no CUDA call) takes its device's primary one.  False if it cannot be had.
bool here(int* device, unsigned long long* context) {
  if (cudaGetDevice(device) != cudaSuccess) return false;
  if (current_context_id(context)) return true;
  return cudaSetDevice(*device) == cudaSuccess && current_context_id(context);
}

struct Driver {
  CUresult (*get_current)(CUcontext*);
  CUresult (*set_current)(CUcontext);
  CUresult (*get_id)(CUcontext, unsigned long long*);
  CUresult (*device)(CUdevice*, int);
  CUresult (*primary_state)(CUdevice, unsigned*, int*);
  CUresult (*primary_retain)(CUcontext*, CUdevice);
  CUresult (*primary_release)(CUdevice);
  bool complete;
};
template <typename F>
bool entry(F* f, const char* name, int version) {
  *f = reinterpret_cast<F>(driver_entry(name, version));
  return *f != nullptr;
}
const Driver& driver() {
  static const Driver d = [] {
    Driver v{};
    v.complete = entry(&v.get_current, "cuCtxGetCurrent", 4000) && entry(&v.set_current, "cuCtxSetCurrent", 4000) &&
                 entry(&v.get_id, "cuCtxGetId", 12000) && entry(&v.device, "cuDeviceGet", 2000) &&
                 entry(&v.primary_state, "cuDevicePrimaryCtxGetState", 7000) &&
                 entry(&v.primary_retain, "cuDevicePrimaryCtxRetain", 7000) &&
                 entry(&v.primary_release, "cuDevicePrimaryCtxRelease", 11000);
    return v;
  }();
  return d;
}

// A device's primary context: its identifier, none (no such context exists now), or not known.
enum Primary { kUnknown, kNone, kHave };
Primary primary_context(int device, unsigned long long* id) {
  const Driver& d = driver();
  CUdevice dev;
  unsigned flags;
  int active = 0;
  if (!d.complete || d.device(&dev, device) != CUDA_SUCCESS || d.primary_state(dev, &flags, &active) != CUDA_SUCCESS)
    return kUnknown;
  if (!active) return kNone;
  CUcontext ctx = nullptr;
  if (d.primary_retain(&ctx, dev) != CUDA_SUCCESS) return kUnknown;
  const bool ok = d.get_id(ctx, id) == CUDA_SUCCESS;
  d.primary_release(dev);
  return ok ? kHave : kUnknown;
}

// Free blocks of the cache, the oldest first, until at most `most` bytes are left in it; only blocks
// of device `only` unless that is negative.  A block that cannot be freed stays.
void shrink(size_t most, int only) {
  int device = 0;
  CUcontext caller = nullptr;
  bool entered = false;
  for (auto it = g_cached.begin(); it != g_cached.end() && g_cached_bytes > most;) {
    unsigned long long id = 0;
    const Primary p = only >= 0 && it->device != only ? kUnknown : primary_context(it->device, &id);
    if (p == kUnknown) {
      ++it;
      continue;
    }
    if (p == kHave && id == it->context) {
      if (!entered) {
        if (cudaGetDevice(&device) != cudaSuccess || driver().get_current(&caller) != CUDA_SUCCESS) return;
        entered = true;
      }
      if (cudaSetDevice(it->device) != cudaSuccess || cudaFree(it->ptr) != cudaSuccess) {
        cudaGetLastError();
        ++it;
        continue;
      }
    }
    g_cached_bytes -= it->bytes;
    it = g_cached.erase(it);
  }
  if (entered) {
    cudaSetDevice(device);
    if (caller) driver().set_current(caller);
  }
}

// alloc(), once more if it found no memory and blocks of this device could be given back (under the
// mutex).
template <typename F>
cudaError_t retried(F alloc) {
  const cudaError_t e = alloc();
  if (e != cudaErrorMemoryAllocation) return e;
  int device = 0;
  unsigned long long context = 0;
  const size_t kept = g_cached_bytes;
  if (kept > 0 && here(&device, &context)) shrink(0, device);
  if (g_cached_bytes == kept) return e;
  cudaGetLastError();
  return alloc();
}

}  // namespace

cudaError_t device_malloc(void** out, size_t bytes) {
  std::lock_guard<std::mutex> lock(g_mutex);
  return retried([&] { return cudaMalloc(out, bytes); });
}

cudaError_t device_malloc_async(void** out, size_t bytes, cudaStream_t s) {
  std::lock_guard<std::mutex> lock(g_mutex);
  return retried([&] { return cudaMallocAsync(out, bytes, s); });
}

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
    const cudaError_t e = retried([&] { return cudaMalloc(out, bytes); });
    if (e != cudaSuccess) {
      *out = nullptr;
      return e;
    }
    if (known) g_in_use[*out] = Block{*out, bytes, device, context};
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
    unsigned long long primary = 0;
    if (idle && b.bytes <= kMaxCached && here(&device, &context) && b.device == device && b.context == context &&
        primary_context(device, &primary) == kHave && primary == context) {
      shrink(kMaxCached - b.bytes, -1);
      try {
        if (g_cached_bytes + b.bytes <= kMaxCached) {
          g_cached.push_back(b);
          g_cached_bytes += b.bytes;
          return;
        }
      } catch (const std::bad_alloc&) {
      }
    }
  }
  cudaFree(ptr);
}

}  // namespace lbmhd_gpu

extern "C" void lbmhd_release_cached_memory(void) {
  std::lock_guard<std::mutex> lock(lbmhd_gpu::g_mutex);
  lbmhd_gpu::shrink(0, -1);
}
