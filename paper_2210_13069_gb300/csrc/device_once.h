// device_once.h -- what a launch needs to know or set once per device, not once per process.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

namespace lrtei {

constexpr int kMaxDevices = 64;  // remembered ones; others are asked at every launch

// Opts KERNEL in to `bytes` of dynamic shared memory (beyond 48 KB a launch is refused otherwise) on the current device:
// the attribute belongs to the device.  Remembered, so that launches inside a stream capture make no other calls.
template <auto KERNEL>
cudaError_t shared_opt_in(size_t bytes) {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const uint64_t bit = dev < kMaxDevices ? 1ULL << dev : 0;
  if (done.load() & bit) return cudaSuccess;
  e = cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) done.fetch_or(bit);
  return e;
}

// SMs of the current device.
inline cudaError_t sm_count(int* n) {
  static std::atomic<int> known[kMaxDevices];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  *n = dev < kMaxDevices ? known[dev].load() : 0;
  if (*n > 0) return cudaSuccess;
  e = cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && dev < kMaxDevices) known[dev].store(*n);
  return e;
}

}  // namespace lrtei
