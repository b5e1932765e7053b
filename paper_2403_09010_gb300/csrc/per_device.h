// Host-side settings that CUDA keeps per device and kernel.
#pragma once

#include <cuda_runtime_api.h>
#include <stdint.h>

#include <atomic>

namespace xtn {

// Runs a setting once on each device it is needed on: a kernel's shared-memory
// limit is the current device's alone, so a process that goes on to a second
// device sets it there as well.  One static object per kernel; a setting that
// failed is tried again by the next call (and the launch behind it reports).
class PerDevice {
 public:
  template <class F>
  void operator()(F&& set) {
    int dev = -1;
    const bool known = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64;
    const uint64_t bit = known ? (uint64_t)1 << dev : 0;
    if (bit & done_.load(std::memory_order_acquire)) return;
    if (set() == cudaSuccess && known) done_.fetch_or(bit, std::memory_order_release);
  }

 private:
  std::atomic<uint64_t> done_{0};
};

// Lets a kernel's blocks take `bytes` of dynamic shared memory; all: the SM's
// memory that serves as L1 or shared goes to shared as far as it may.
inline cudaError_t allow_shared(const void* kernel, int bytes, bool all = true) {
  const cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess || !all) return e;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
}

}  // namespace xtn
