// Something to be done once on every device that a process uses, such as a kernel's
// opt-in to large dynamic shared memory, which cudaFuncSetAttribute grants on the
// current device only.
#pragma once

#include <mutex>
#include <set>

#include "common.cuh"

namespace dfjk {

class OncePerDevice {
  std::mutex mu;
  std::set<int> done;

 public:
  // Runs `f` unless it has run on the current device before (one that threw has not).
  template <class F>
  void operator()(F f) {
    int dev = 0;
    DFJK_CUDA_CHECK(cudaGetDevice(&dev));
    std::lock_guard<std::mutex> lk(mu);
    if (done.count(dev)) return;
    f();
    done.insert(dev);
  }
};

// Dynamic shared memory of `kernel` raised to `bytes` (one object per kernel).
template <class K>
void allow_smem(OncePerDevice &once, K *kernel, int bytes) {
  const void *f = reinterpret_cast<const void *>(kernel);
  once([&] { DFJK_CUDA_CHECK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes)); });
}

}  // namespace dfjk
