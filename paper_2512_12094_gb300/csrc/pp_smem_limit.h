// The dynamic shared memory a kernel may be launched with.
//
// Above 48 KB it has to be allowed by an attribute that belongs to the kernel on
// the current device, so it is raised once per kernel and device; a refused
// attempt is made again at the next launch.  (A call per launch would do as well;
// a layer of many short phases launches one every few microseconds.)
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <cstdint>

namespace ppk {

// One per kernel, in static storage; used by any number of threads.
class SmemLimit {
 public:
  template <class Kernel>
  cudaError_t raise(Kernel* kernel, size_t bytes) {
    int device = 0;
    cudaError_t e = cudaGetDevice(&device);
    if (e != cudaSuccess) return e;
    const uint64_t bit = device < 64 ? 1ull << device : 0ull;  // beyond: at every launch
    if (raised_.load(std::memory_order_acquire) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) raised_.fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<uint64_t> raised_{0};  // devices it was raised on
};

}  // namespace ppk
