#include "device_scratch.h"

#include <algorithm>
#include <mutex>

namespace pdds {
namespace {

__device__ __align__(256) unsigned char g_scratch[DeviceScratch::kKeep];

std::mutex g_mu;
constexpr int kContexts = 64;
void* g_taken[kContexts] = {};  // the arrays in use, one per context at most

}  // namespace

DeviceScratch::~DeviceScratch() {
  if (!ptr_) return;
  if (!kept_) {
    cudaFree(ptr_);
    return;
  }
  std::lock_guard<std::mutex> lock(g_mu);
  *std::find(g_taken, g_taken + kContexts, ptr_) = nullptr;
}

cudaError_t DeviceScratch::get(size_t bytes) {
  if (bytes <= kKeep) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_scratch);
    if (e != cudaSuccess) return e;
    std::lock_guard<std::mutex> lock(g_mu);
    void** const end = g_taken + kContexts;
    void** const free_slot = std::find(g_taken, end, nullptr);
    if (std::find(g_taken, end, p) == end && free_slot != end) {
      *free_slot = ptr_ = p;
      kept_ = true;
      return cudaSuccess;
    }
  }
  return cudaMalloc(&ptr_, bytes);
}

}  // namespace pdds
