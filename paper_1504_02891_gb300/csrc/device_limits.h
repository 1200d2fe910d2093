// device_limits.h -- launch limits of the current device: kernel attributes and
// occupancies belong to a device, so they are looked up once on each device
// that a process uses.
#pragma once
#include <cuda_runtime_api.h>
#include <stddef.h>
#include <atomic>

namespace gpe {

constexpr int MAX_DEVICES = 64;   // devices whose values are kept (others: looked up on every call)

// Multiprocessors of the current device.
int num_sms();

// Raise a kernel's dynamic shared memory limit on the current device to at
// least `bytes` (never lowered: other threads may be launching it with more).
cudaError_t raise_smem(const void* fn, size_t bytes);

// What a launcher keeps of one kernel and launch shape (a function-local
// static): per device the resident CTAs per SM, 0 where it has not been looked
// up.  A failed lookup is not kept.
struct KernelShape {
  std::atomic<int> occ[MAX_DEVICES];
};
// The shape's resident CTAs per SM (at least 1) on the current device, with the
// shared memory limit raised there.
cudaError_t kernel_shape(KernelShape& shape, const void* fn, int threads, size_t smem, int* occ);

}  // namespace gpe
