// Device memory of one DMRG run, kept between its steps.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

namespace dmrg {

// Spare blocks of a DMRG run: sizes up to 4 MiB in classes a quarter of an
// octave apart (at most a quarter of a block unused; larger arrays come from
// and go back to the driver), at most 64 spare blocks of each, released with
// the run.  A block put back is handed out again at once, so everything that
// uses the pool runs on one stream (the run's, the legacy default stream); a
// run's calls do not overlap.  When the device has no memory left the spare
// blocks are given back and the allocation is tried again.
// `current` is the calling thread's pool, set for the length of a call.
class DevPool {
 public:
  static constexpr int MIN_LOG = 12, MAX_LOG = 22, PER_OCTAVE = 4;
  static constexpr int CLASSES = (MAX_LOG - MIN_LOG) * PER_OCTAVE + 1;
  static constexpr int MAX_KEPT = 64;
  static constexpr size_t capacity(int c) {
    return (size_t)(PER_OCTAVE + c % PER_OCTAVE) << (c / PER_OCTAVE + MIN_LOG - 2);
  }
  void* get(size_t bytes);  // throws std::runtime_error
  void put(void* p, size_t bytes) noexcept;  // bytes: as asked for
  void trim() noexcept;     // give every spare block back
  ~DevPool() { trim(); }
  static DevPool* current();
  static DevPool* set_current(DevPool* p);  // returns the previous one

 private:
  static int size_class(size_t bytes);  // CLASSES: larger than any
  void* free_[CLASSES][MAX_KEPT] = {};
  int n_[CLASSES] = {};
};

// cudaMalloc that gives back the spare blocks of the calling thread's pool
// before it reports that memory has run out
cudaError_t dev_malloc(void** p, size_t bytes);

}  // namespace dmrg
