// Device memory: allocations of the library, and the blocks kept between a handle's tapes.
#include <cuda_runtime.h>

#include <atomic>
#include <set>

#include "internal.h"

namespace lbm {
namespace {

std::atomic<size_t> g_tape_kept{0};  // bytes kept by all handles

// Every handle's TapeMemory.  Never destroyed: handles may outlive static objects.  Its lock is taken before a
// TapeMemory's, never after.
struct Registry {
  std::mutex mu;
  std::set<TapeMemory*> all;
};
Registry& registry() {
  static Registry* const r = new Registry;
  return *r;
}

}  // namespace

cudaError_t device_alloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    Registry& r = registry();
    {
      std::lock_guard<std::mutex> lock(r.mu);
      for (TapeMemory* m : r.all) m->release();
    }
    e = cudaMalloc(p, bytes);
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
  }
  return e;
}

TapeMemory::TapeMemory() {
  Registry& r = registry();
  std::lock_guard<std::mutex> lock(r.mu);
  r.all.insert(this);
}

TapeMemory::~TapeMemory() {
  Registry& r = registry();
  std::lock_guard<std::mutex> lock(r.mu);
  r.all.erase(this);
}

void* TapeMemory::take(size_t need, size_t* got) {
  {
    std::lock_guard<std::mutex> lock(mu);
    if (mem && bytes >= need && bytes / 2 <= need) {
      void* const m = mem;
      *got = bytes;
      g_tape_kept -= bytes;
      mem = nullptr;
      bytes = 0;
      return m;
    }
  }
  release();
  void* m = nullptr;
  *got = need;
  return device_alloc(&m, need) == cudaSuccess ? m : nullptr;
}

bool TapeMemory::give(void* m, size_t size) {
  std::lock_guard<std::mutex> lock(mu);
  if (closed || mem) return false;
  if ((g_tape_kept += size) > kTapeKeepTotal) {
    g_tape_kept -= size;
    return false;
  }
  mem = m;
  bytes = size;
  return true;
}

void TapeMemory::release() {
  std::lock_guard<std::mutex> lock(mu);
  if (!mem) return;
  cudaFree(mem);
  g_tape_kept -= bytes;
  mem = nullptr;
  bytes = 0;
}

void TapeMemory::close() {
  {
    std::lock_guard<std::mutex> lock(mu);
    closed = true;
  }
  release();
}

}  // namespace lbm
