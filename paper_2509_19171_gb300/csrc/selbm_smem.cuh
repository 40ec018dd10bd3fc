// Dynamic shared-memory limit of a kernel.
//
// The limit belongs to the function on its device, not to a launch or a thread, and setting a lower
// one takes the higher away.  Launches of one kernel differ in size (walls of an element, elements
// of a CTA, order), so each kernel gets the most that its static share leaves, once per device:
// whatever other threads launch, none lowers it.  A launch takes what it asks for, not the limit.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace slb {

// K: the kernel, as a template value (one record per kernel)
template <auto K>
cudaError_t raise_smem(size_t smem) {
  static std::atomic<unsigned long long> done{0};        // devices whose limit is set
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
  if (done.load(std::memory_order_acquire) & bit) return cudaSuccess;
  int most = 0;
  cudaFuncAttributes fa{};
  if ((e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) return e;
  if ((e = cudaFuncGetAttributes(&fa, K)) != cudaSuccess) return e;
  const int limit = most - (int)fa.sharedSizeBytes;
  if ((size_t)(limit > 0 ? limit : 0) < smem) return cudaErrorInvalidValue;
  if ((e = cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, limit)) != cudaSuccess) return e;
  done.fetch_or(bit, std::memory_order_release);
  return cudaSuccess;
}

}  // namespace slb
