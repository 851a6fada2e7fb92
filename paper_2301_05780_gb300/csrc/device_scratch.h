// Small device scratch of the context-free network calls (pdds_mlp_train,
// pdds_mlp_eval and their tensor-core forms), which synchronize before they
// return.  cudaMalloc and cudaFree synchronize the device and cost about 0.15
// ms a call, a third of a 1.6e6-point evaluation, so one buffer per device is
// kept between calls: at most kKeep bytes, handed to one call at a time (a
// call that finds it taken, or needs more, allocates its own), and looked at
// before each use, so that a device reset in between only drops it.
#pragma once
#include <cuda_runtime.h>

#include <mutex>

namespace pdds {

class DeviceScratch {
 public:
  static constexpr size_t kKeep = 1 << 20;
  DeviceScratch() = default;
  DeviceScratch(const DeviceScratch&) = delete;
  DeviceScratch& operator=(const DeviceScratch&) = delete;
  // After the work that uses the buffer has been synchronized with.
  ~DeviceScratch() {
    if (!ptr_) return;
    if (!kept_) {
      cudaFree(ptr_);
      return;
    }
    std::lock_guard<std::mutex> lock(mutex());
    slot(dev_).taken = false;
  }
  cudaError_t get(size_t bytes) {
    cudaError_t e = cudaGetDevice(&dev_);
    if (e != cudaSuccess) return e;
    if (bytes <= kKeep && dev_ >= 0 && dev_ < kDevices) {
      std::lock_guard<std::mutex> lock(mutex());
      Slot& s = slot(dev_);
      if (!s.taken) {
        if (s.ptr) {
          cudaPointerAttributes a;
          const cudaError_t q = cudaPointerGetAttributes(&a, s.ptr);
          if (q != cudaSuccess || a.type != cudaMemoryTypeDevice || a.device != dev_) {
            (void)cudaGetLastError();
            s.ptr = nullptr;  // the context it belonged to is gone
          }
        }
        if (!s.ptr && (e = cudaMalloc(&s.ptr, kKeep)) != cudaSuccess) {
          s.ptr = nullptr;
          return e;
        }
        s.taken = kept_ = true;
        ptr_ = s.ptr;
        return cudaSuccess;
      }
    }
    return cudaMalloc(&ptr_, bytes);
  }
  void* ptr() const { return ptr_; }

 private:
  struct Slot {
    void* ptr = nullptr;
    bool taken = false;
  };
  static constexpr int kDevices = 64;
  static std::mutex& mutex() {
    static std::mutex m;
    return m;
  }
  static Slot& slot(int dev) {
    static Slot s[kDevices];
    return s[dev];
  }
  void* ptr_ = nullptr;
  int dev_ = 0;
  bool kept_ = false;
};

}  // namespace pdds
