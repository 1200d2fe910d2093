// device_limits.cu -- see device_limits.h (host code only).
#include "device_limits.h"
#include <map>
#include <mutex>
#include <utility>

namespace gpe {

static int current_device() {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess ? dev : 0;
}

int num_sms() {
  static std::atomic<int> sms[MAX_DEVICES];
  const int dev = current_device();
  const bool kept = dev >= 0 && dev < MAX_DEVICES;
  int n = kept ? sms[dev].load(std::memory_order_relaxed) : 0;
  if (n > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 152;
  if (kept) sms[dev].store(n, std::memory_order_relaxed);
  return n;
}

cudaError_t raise_smem(const void* fn, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, size_t> allowed;   // (device, kernel)
  const int dev = current_device();
  std::lock_guard<std::mutex> lk(mu);
  const auto it = allowed.find({dev, fn});
  if (it != allowed.end() && bytes <= it->second) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) allowed[{dev, fn}] = bytes;
  return e;
}

cudaError_t kernel_shape(KernelShape& shape, const void* fn, int threads, size_t smem, int* occ) {
  const int dev = current_device();
  const bool kept = dev >= 0 && dev < MAX_DEVICES;
  int n = kept ? shape.occ[dev].load(std::memory_order_acquire) : 0;
  if (n < 1) {
    cudaError_t e = raise_smem(fn, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, threads, smem);
    if (e != cudaSuccess) return e;
    if (n < 1) n = 1;
    if (kept) shape.occ[dev].store(n, std::memory_order_release);
  }
  *occ = n;
  return cudaSuccess;
}

}  // namespace gpe
