// Spare device memory of a DMRG run (devpool.h); host code only.
#include "devpool.h"

#include <stdexcept>
#include <string>

namespace dmrg {

namespace {
thread_local DevPool* g_pool = nullptr;
}  // namespace

DevPool* DevPool::current() { return g_pool; }
DevPool* DevPool::set_current(DevPool* p) {
  DevPool* old = g_pool;
  g_pool = p;
  return old;
}

int DevPool::size_class(size_t bytes) {
  int c = 0;
  while (c < CLASSES && capacity(c) < bytes) ++c;
  return c;
}

void* DevPool::get(size_t bytes) {
  const int c = size_class(bytes);
  if (c < CLASSES && n_[c] > 0) return free_[c][--n_[c]];
  const size_t want = c < CLASSES ? capacity(c) : bytes;
  void* p = nullptr;
  cudaError_t e = cudaMalloc(&p, want);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    trim();
    e = cudaMalloc(&p, want);
  }
  if (e != cudaSuccess) throw std::runtime_error(std::string("cudaMalloc: ") + cudaGetErrorString(e));
  return p;
}

void DevPool::put(void* p, size_t bytes) noexcept {
  const int c = size_class(bytes);
  if (c < CLASSES && n_[c] < MAX_KEPT) free_[c][n_[c]++] = p;
  else cudaFree(p);
}

void DevPool::trim() noexcept {
  for (int c = 0; c < CLASSES; ++c) {
    while (n_[c] > 0) cudaFree(free_[c][--n_[c]]);
  }
}

cudaError_t dev_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  DevPool* pool = DevPool::current();
  if (e != cudaErrorMemoryAllocation || !pool) return e;
  cudaGetLastError();
  pool->trim();
  return cudaMalloc(p, bytes);
}

}  // namespace dmrg
