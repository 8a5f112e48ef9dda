"""The bookkeeping of device memory kept from freed handles, on the CPU: lbmhd_memory.cu compiled
against a stand-in for the CUDA runtime and driver that has two small devices, a current device and
context per thread, a primary context per device that a reset replaces, and contexts of the driver API."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1705_09807_gb300", "csrc")

STAND_IN = r"""
#include <cstdio>
#include <cstring>
#include <map>
#include <thread>
#include "lbmhd_memory.h"
#include <cuda.h>

struct Ctx { int device; unsigned long long id; };
static unsigned long long next_id = 1;
static Ctx primary_ctx[2];
static bool active[2];
struct Mem { size_t bytes; int device; unsigned long long id; };
static std::map<void*, Mem> mem;
static size_t capacity[2] = {(size_t)4 << 30, (size_t)4 << 30};
static int wrong_frees = 0;
static thread_local int cur_device = 0;
static thread_local Ctx* cur = nullptr;

static size_t used(int device) {
  size_t s = 0;
  for (auto& m : mem) if (m.second.device == device) s += m.second.bytes;
  return s;
}
static void need_primary(int d) { if (!active[d]) { primary_ctx[d] = Ctx{d, next_id++}; active[d] = true; } }
static void bind() { if (!cur) { need_primary(cur_device); cur = &primary_ctx[cur_device]; } }
static void reset(int d) {
  for (auto it = mem.begin(); it != mem.end();) it = it->second.id == primary_ctx[d].id ? mem.erase(it) : std::next(it);
  active[d] = false;
  if (cur == &primary_ctx[d]) cur = nullptr;
}
extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = cur ? cur->device : cur_device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { cur_device = d; need_primary(d); cur = &primary_ctx[d]; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) {
  bind();
  if (used(cur->device) + n > capacity[cur->device]) return cudaErrorMemoryAllocation;
  static char* at = (char*)0x1000;
  *p = at; at += 0x1000;
  mem[*p] = Mem{n, cur->device, cur->id};
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  bind();
  auto it = mem.find(p);
  if (it == mem.end() || it->second.id != cur->id) { ++wrong_frees; return cudaErrorInvalidValue; }
  mem.erase(it);
  return cudaSuccess;
}
}
static CUresult get_current(CUcontext* c) { *c = (CUcontext)cur; return CUDA_SUCCESS; }
static CUresult set_current(CUcontext c) { cur = (Ctx*)c; if (cur) cur_device = cur->device; return CUDA_SUCCESS; }
static CUresult get_id(CUcontext c, unsigned long long* id) { *id = ((Ctx*)c)->id; return CUDA_SUCCESS; }
static CUresult device_get(CUdevice* d, int n) { *d = n; return CUDA_SUCCESS; }
static CUresult state(CUdevice d, unsigned* f, int* a) { *f = 0; *a = active[d]; return CUDA_SUCCESS; }
static CUresult retain(CUcontext* c, CUdevice d) { need_primary(d); *c = (CUcontext)&primary_ctx[d]; return CUDA_SUCCESS; }
static CUresult release(CUdevice) { return CUDA_SUCCESS; }
namespace lbmhd_gpu {
void* driver_entry(const char* n, int) {
  if (!strcmp(n, "cuCtxGetCurrent")) return (void*)get_current;
  if (!strcmp(n, "cuCtxSetCurrent")) return (void*)set_current;
  if (!strcmp(n, "cuCtxGetId")) return (void*)get_id;
  if (!strcmp(n, "cuDeviceGet")) return (void*)device_get;
  if (!strcmp(n, "cuDevicePrimaryCtxGetState")) return (void*)state;
  if (!strcmp(n, "cuDevicePrimaryCtxRetain")) return (void*)retain;
  if (!strcmp(n, "cuDevicePrimaryCtxRelease")) return (void*)release;
  return nullptr;
}
bool current_context_id(unsigned long long* id) { if (!cur) return false; *id = cur->id; return true; }
}
extern "C" void lbmhd_release_cached_memory(void);
using namespace lbmhd_gpu;
static const size_t MiB = (size_t)1 << 20;
static int failures = 0;
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); ++failures; } } while (0)
static void* keep(size_t n) { void* p = nullptr; CHECK(device_alloc(&p, n) == cudaSuccess); device_free(p, true); return p; }
"""

CASES = {
    # a thread that has made no CUDA call returns the memory; so does one on another device
    "release_from_other_threads": r"""
  keep(300 * MiB);
  CHECK(used(0) == 300 * MiB);
  std::thread([] { lbmhd_release_cached_memory(); }).join();
  CHECK(used(0) == 0);
  keep(300 * MiB);
  std::thread([] { cudaSetDevice(1); keep(200 * MiB); lbmhd_release_cached_memory();
                   int d; cudaGetDevice(&d); CHECK(d == 1); CHECK(cur == &primary_ctx[1]); }).join();
  CHECK(used(0) == 0 && used(1) == 0);
""",
    # a new thread's allocation finds the kept block
    "reuse_in_a_new_thread": r"""
  void* p = keep(300 * MiB);
  std::thread([p] { void* q = nullptr; CHECK(device_alloc(&q, 300 * MiB) == cudaSuccess); CHECK(q == p); device_free(q, true); }).join();
  CHECK(used(0) == 300 * MiB);
""",
    # a reset takes the blocks with it: forgotten, never freed; the account is clear again
    "reset_context": r"""
  keep(900 * MiB);
  reset(0);
  void* p = keep(800 * MiB);
  CHECK(used(0) == 800 * MiB);
  void* q = nullptr;
  CHECK(device_alloc(&q, 800 * MiB) == cudaSuccess && q == p);
  device_free(q, true);
  reset(0);
  lbmhd_release_cached_memory();
  CHECK(!active[0]);
""",
    # blocks of a context of the driver API are not kept: nothing could tell later whether it lives
    "driver_context": r"""
  keep(100 * MiB);
  Ctx own{0, next_id++};
  set_current((CUcontext)&own);
  keep(200 * MiB);
  CHECK(used(0) == 100 * MiB);
  lbmhd_release_cached_memory();
  CHECK(used(0) == 0 && cur == &own);
""",
    # the bound holds over all devices, the oldest blocks go first
    "bound": r"""
  keep(600 * MiB);
  cudaSetDevice(1);
  keep(400 * MiB);
  CHECK(used(0) + used(1) == 1000 * MiB);
  keep(300 * MiB);
  CHECK(used(0) == 0 && used(1) == 700 * MiB);
  int d; cudaGetDevice(&d); CHECK(d == 1);
  keep(1100 * MiB);
  CHECK(used(1) == 700 * MiB);
""",
    # an allocation that fails gets the kept blocks of its device, and then the error if that is not enough
    "out_of_memory": r"""
  capacity[0] = 1000 * MiB;
  keep(600 * MiB);
  void* p = nullptr;
  CHECK(device_alloc(&p, 700 * MiB) == cudaSuccess);
  CHECK(used(0) == 700 * MiB);
  void* q = nullptr;
  CHECK(device_alloc(&q, 400 * MiB) == cudaErrorMemoryAllocation && !q);
  device_free(p, false);
  CHECK(used(0) == 0);
""",
    # the library's other allocations get them as well, those of their own device
    "out_of_memory_elsewhere": r"""
  capacity[0] = capacity[1] = 1000 * MiB;
  for (int async = 0; async < 2; ++async) {
    keep(600 * MiB);
    cudaSetDevice(1);
    keep(100 * MiB);
    cudaSetDevice(0);
    void* p = nullptr;
    CHECK((async ? device_malloc_async(&p, 700 * MiB, nullptr) : device_malloc(&p, 700 * MiB)) == cudaSuccess);
    CHECK(used(0) == 700 * MiB && used(1) == 100 * MiB);
    cudaFree(p);
  }
  void* q = nullptr;
  CHECK(device_malloc(&q, 1100 * MiB) == cudaErrorMemoryAllocation);
""",
}


@pytest.fixture(scope="module")
def include_dir():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda.h")):
        inc = "/usr/local/cuda/include"
    return inc


@pytest.mark.parametrize("case", sorted(CASES))
def test_memory_of_freed_handles(case, tmp_path, include_dir):
    main = tmp_path / "main.cpp"
    main.write_text(STAND_IN + "int main() {" + CASES[case] +
                    "  CHECK(wrong_frees == 0);\n  return failures;\n}\n")
    exe = str(tmp_path / "main")
    cmd = ["g++", "-std=c++17", "-O1", "-o", exe, str(main), "-x", "c++", os.path.join(CSRC, "lbmhd_memory.cu"),
           "-I", CSRC, "-I", os.path.join(ROOT, "include"), "-I", include_dir, "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_every_allocation_can_have_the_kept_memory():
    """No source file but lbmhd_memory.cu calls the runtime's allocation functions itself."""
    import re
    for f in sorted(os.listdir(CSRC)):
        if f != "lbmhd_memory.cu" and os.path.isfile(os.path.join(CSRC, f)):
            with open(os.path.join(CSRC, f)) as fh:
                code = re.sub(r"//[^\n]*", "", fh.read())
            assert not re.search(r"\bcudaMalloc(Async|Managed|Pitch)?\s*\(", code), f
