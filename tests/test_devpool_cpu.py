"""The spare device memory of a DMRG run (csrc/devpool.cu), compiled for the
host against a fake of the CUDA allocator with a limited memory: what it keeps
is bounded, is given back when memory runs out, and is released at the end."""
import os
import shutil
import subprocess

import pytest

from paper_0902_3185_gb300 import build

DRIVER = r"""
#include "devpool.h"

#include <cassert>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <stdexcept>
#include <vector>

static size_t limit = 0, used = 0;
static cudaError_t last = cudaSuccess;
static std::map<void*, size_t> live;

extern "C" cudaError_t cudaMalloc(void** p, size_t n) {
  if (used + n > limit) return last = cudaErrorMemoryAllocation;
  *p = malloc(1);
  live[*p] = n;
  used += n;
  return cudaSuccess;
}
extern "C" cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  assert(live.count(p));
  used -= live[p];
  live.erase(p);
  free(p);
  return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
extern "C" const char* cudaGetErrorString(cudaError_t) { return "out of memory"; }

using namespace dmrg;

int main() {
  const size_t MiB = 1 << 20;
  limit = 1000 * MiB;
  {  // at most a quarter of a block is unused, whatever is asked for; large arrays take what they ask for
    DevPool pool;
    std::vector<std::pair<void*, size_t>> got;
    for (size_t n : {1ul, 4096ul, 4097ul, 5120ul, 100000ul, MiB, MiB + 1, 3 * MiB + 5, 4 * MiB, 4 * MiB + 1, 9 * MiB}) {
      const size_t before = used;
      void* p = pool.get(n);
      const size_t took = used - before;
      assert(took >= n && (took <= 4096 || 4 * took <= 5 * n + 4096));
      if (n > 4 * MiB) assert(took == n);
      got.push_back({p, n});
    }
    for (auto& g : got) pool.put(g.first, g.second);
    // a block put back serves the next request of its class
    const size_t before = used;
    void* p = pool.get(3 * MiB + 1);
    void* q = pool.get(100000);
    assert(used == before);
    pool.put(p, 3 * MiB + 1);
    pool.put(q, 100000);
  }
  assert(used == 0);
  {  // no more than MAX_KEPT spare blocks of a class
    DevPool pool;
    std::vector<void*> v;
    for (int i = 0; i < DevPool::MAX_KEPT + 9; ++i) v.push_back(pool.get(5000));
    for (void* p : v) pool.put(p, 5000);
    assert(live.size() == (size_t)DevPool::MAX_KEPT);
  }
  assert(used == 0);
  {  // memory runs out while blocks are spare: they are given back
    DevPool pool;
    std::vector<void*> v;
    for (int i = 0; i < 50; ++i) v.push_back(pool.get(4 * MiB));
    for (void* p : v) pool.put(p, 4 * MiB);
    assert(used == 200 * MiB);
    void* big = pool.get(900 * MiB);
    assert(used == 900 * MiB);
    pool.put(big, 900 * MiB);
    assert(used == 0);
  }
  {  // the same for an allocation beside the pool, in a call of the pool's run only
    DevPool pool;
    pool.put(pool.get(4 * MiB), 4 * MiB);
    void* p = nullptr;
    assert(dev_malloc(&p, 998 * MiB) == cudaErrorMemoryAllocation);
    DevPool* old = DevPool::set_current(&pool);
    assert(old == nullptr);
    assert(dev_malloc(&p, 998 * MiB) == cudaSuccess);
    assert(dev_malloc(&p, 998 * MiB) == cudaErrorMemoryAllocation);
    assert(cudaGetLastError() == cudaErrorMemoryAllocation);  // what tells the caller the reason
    cudaFree(p);
    DevPool::set_current(old);
    bool thrown = false;
    try { pool.get(2000 * MiB); } catch (const std::runtime_error&) { thrown = true; }
    assert(thrown && cudaGetLastError() == cudaErrorMemoryAllocation);
  }
  assert(used == 0);
  puts("ok");
}
"""


def test_pool_is_bounded_and_given_back(tmp_path):
    cxx = shutil.which("g++")
    include = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")
    if not cxx or not os.path.exists(os.path.join(include, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    (tmp_path / "driver.cpp").write_text(DRIVER)
    exe = str(tmp_path / "driver")
    subprocess.run([cxx, "-std=c++17", "-O1", "-I" + build.CSRC, "-I" + include, "-x", "c++",
                    os.path.join(build.CSRC, "devpool.cu"), str(tmp_path / "driver.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.stdout.strip() == "ok", out.stdout + out.stderr
