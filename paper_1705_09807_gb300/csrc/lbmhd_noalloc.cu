// Diagnostics of caller-provided device moment fields without any device allocation.
//
// Some callers cannot call cudaMalloc: code that runs inside another framework's memory
// pool or arena (every byte must come from it), code running under a strict memory budget
// that forbids new allocations after start-up, or code on a path where an allocation would
// synchronise the device.  This entry point serves them: the caller passes its device
// inputs and output, and the per-block partial sums live in a fixed, file-scope device
// array of this library instead of a buffer allocated per call.
//
// The reduction is the same as lbmhd_diagnostics' (sums, maxima and the instability flag),
// by the same kernels (lbmhd_diag.cuh), combined in a fixed order, so the result is bitwise
// reproducible for a given grid.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdio>
#include <mutex>

#include "lbmhd.h"
#include "lbmhd_diag.cuh"
#include "lbmhd_internal.cuh"

using namespace lbmhd_gpu;

namespace {

constexpr long kCellsPerBlock = 4096;
constexpr int kMaxBlocks = 4096;       // capacity: 4096 x 4096 = 16,777,216 cells
constexpr int kSlots = kDiagSlots;     // the public values plus the instability flag
constexpr int kMaxDevices = 64;

// Partial results, one record of kSlots doubles per block: 4096 x 11 x 8 B = 352 KiB held on
// every GPU that loads the library, until the process exits.  Every call overwrites the
// records it reads, so nothing has to be cleared between calls.
static __device__ __align__(256) double g_partials[kMaxBlocks * kSlots];

std::mutex g_setup_mutex;

int set_error(int code, const char* msg) {
  lbmhd_gpu::set_thread_error(msg);
  return code;
}

}  // namespace

void* lbmhd_gpu::driver_entry(const char* name, int version) {
  void* f = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion(name, &f, version, cudaEnableDefault, &q) != cudaSuccess ||
      q != cudaDriverEntryPointSuccess)
    return nullptr;
  return f;
}

// Identifier of the calling thread's current context; false if it cannot be had (no current
// context yet, or a driver without cuCtxGetId), in which case the caller looks the address up
// afresh.  cuCtxGetId gives a context an identifier that is unique for the life of the process, so
// a context that was destroyed and re-created (for example after cudaDeviceReset) is told apart
// from its predecessor even if its handle value is reused.
bool lbmhd_gpu::current_context_id(unsigned long long* id) {
  using CtxGetCurrentFn = CUresult (*)(CUcontext*);
  using CtxGetIdFn = CUresult (*)(CUcontext, unsigned long long*);
  static const auto get_current = reinterpret_cast<CtxGetCurrentFn>(driver_entry("cuCtxGetCurrent", 4000));
  static const auto get_id = reinterpret_cast<CtxGetIdFn>(driver_entry("cuCtxGetId", 12000));
  if (!get_current || !get_id) return false;
  CUcontext ctx = nullptr;
  if (get_current(&ctx) != CUDA_SUCCESS || !ctx) return false;
  return get_id(ctx, id) == CUDA_SUCCESS;
}

namespace {

struct PartialsAddr {
  double* ptr = nullptr;
  unsigned long long ctx_id = 0;
};
PartialsAddr g_partials_addr[kMaxDevices];

// Device address of g_partials in the current device's current context.  It is looked up with
// cudaGetSymbolAddress on the first call in a context (which also loads the library's module
// into that context if it is not loaded yet) and cached with the context's identifier; a call
// in another context -- a different device, or the same device after its primary context was
// reset -- looks it up again instead of using a stale address.
int partials_address(double** out) {
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return set_error(LBMHD_ERR_CUDA, cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return set_error(LBMHD_ERR_INVALID, "device ordinal out of range");
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  unsigned long long id = 0;
  const bool have_id = current_context_id(&id);
  PartialsAddr& a = g_partials_addr[dev];
  if (!(have_id && a.ptr && a.ctx_id == id)) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_partials);
    if (e != cudaSuccess || !p) {
      char buf[256];
      snprintf(buf, sizeof buf, "cudaGetSymbolAddress of the diagnostics scratch failed: %s",
               cudaGetErrorString(e));
      return set_error(LBMHD_ERR_CUDA, buf);
    }
    a.ptr = static_cast<double*>(p);
    // the lookup above makes the primary context current if it was not yet
    a.ctx_id = current_context_id(&id) ? id : 0;
  }
  *out = a.ptr;
  return LBMHD_OK;
}

}  // namespace

extern "C" int lbmhd_diagnostics_fields_noalloc(const double* rho, const double* ux,
                                                const double* uy, const double* bx,
                                                const double* by, int nx, int ny, double* out,
                                                void* stream) {
  if (!rho || !ux || !uy || !bx || !by || !out)
    return set_error(LBMHD_ERR_INVALID, "a field or output pointer is NULL");
  if (nx < 3 || ny < 3) return set_error(LBMHD_ERR_INVALID, "grid sides must be >= 3");
  const long long ncell = (long long)nx * ny;
  if (ncell > (long long)kMaxBlocks * kCellsPerBlock) {
    char buf[256];
    snprintf(buf, sizeof buf,
             "grid %d x %d has %lld cells; the allocation-free diagnostics handle at most %lld",
             nx, ny, ncell, (long long)kMaxBlocks * kCellsPerBlock);
    return set_error(LBMHD_ERR_INVALID, buf);
  }
  double* partials = nullptr;
  int rc = partials_address(&partials);
  if (rc) return rc;
  // a quarter of the records fills the GPU; every record read is written first
  const DiagTiles t = diag_tiles(nx, ny, kMaxBlocks / 4, true, kDiagMinRows);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  launch_diag_partials(rho, ux, uy, bx, by, nx, ny, t, partials, s);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) {
    diag_final_kernel<<<1, 32 * kDiagSlots, 0, s>>>(partials, t.blocks, out);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return set_error(LBMHD_ERR_CUDA, cudaGetErrorString(e));
  return LBMHD_OK;
}
