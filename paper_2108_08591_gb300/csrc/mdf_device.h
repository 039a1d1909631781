// What the library keeps per GPU.
#pragma once

#include <cuda_runtime_api.h>

#include <mutex>

namespace mdf {

constexpr int kMaxDevices = 64;  // ordinals beyond are served without keeping anything

// A step that has to succeed once on every device, such as raising a kernel's
// limits: cudaFuncSetAttribute acts on the current device alone, so a function
// static would leave every other GPU of the process without it.  A failed step
// is tried again by the next call.
class OncePerDevice {
 public:
  template <class Step> cudaError_t operator()(Step step) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return step();
    std::lock_guard<std::mutex> lock(mu_);
    if (done_[dev]) return cudaSuccess;
    const cudaError_t s = step();
    done_[dev] = s == cudaSuccess;
    return s;
  }

 private:
  std::mutex mu_;
  bool done_[kMaxDevices] = {};
};

// A kernel may use up to `bytes` of dynamic shared memory on the current device.
template <class Kernel> cudaError_t allow_smem(OncePerDevice &once, Kernel kernel, size_t bytes) {
  return once([&] { return cudaFuncSetAttribute((const void *)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes); });
}

}  // namespace mdf
