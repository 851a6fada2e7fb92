// Small device scratch of the context-free network calls (pdds_mlp_train,
// pdds_mlp_eval and their tensor-core forms), which synchronize before they
// return.  cudaMalloc and cudaFree synchronize the device and cost about 0.15
// ms a call, a third of a 1.6e6-point evaluation, so calls that need at most
// kKeep bytes take turns on a static device array of that size; a call that
// finds it taken, or needs more, allocates its own.  The array is part of the
// library's image in each CUDA context: its address is asked for at every use,
// so it is always memory of the current context and of nobody else, also after
// a device reset or in a second context of the same device.
#pragma once
#include <cuda_runtime.h>

#include <cstddef>

namespace pdds {

class DeviceScratch {
 public:
  static constexpr size_t kKeep = 1 << 20;
  DeviceScratch() = default;
  DeviceScratch(const DeviceScratch&) = delete;
  DeviceScratch& operator=(const DeviceScratch&) = delete;
  // After the work that uses the buffer has been synchronized with.
  ~DeviceScratch();
  cudaError_t get(size_t bytes);
  void* ptr() const { return ptr_; }

 private:
  void* ptr_ = nullptr;
  bool kept_ = false;
};

}  // namespace pdds
