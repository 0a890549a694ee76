// Opting a kernel in to its dynamic shared memory on the current device, its CTAs per SM there, and the device's SMs.
#pragma once
#include <cuda_runtime.h>

#include <mutex>
#include <unordered_map>

#include "launch_rules.hpp"

namespace pgb {

inline KernelGrants& kernel_grants() {
  static KernelGrants g;
  return g;
}

// Always done (not only above 48 KB): static shared memory counts against the same default limit.  threads > 0: *per_sm
// is the number of CTAs of that size that fit an SM.
template <typename K> inline cudaError_t allow_smem(K kernel, size_t smem, int threads = 0, int* per_sm = nullptr) {
  int dev = 0, n = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const int r = kernel_grants().get(
      dev, reinterpret_cast<const void*>(kernel), smem, threads,
      [&](size_t bytes) {
        return (int)cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
      },
      [&](int* out) { return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kernel, threads, smem); }, &n);
  if (per_sm) *per_sm = n;
  return (cudaError_t)r;
}

// SMs of the current device (0 if it cannot be told).
inline int sm_count() {
  static std::mutex mu;
  static std::unordered_map<int, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(dev);
  if (it != cache.end()) return it->second;
  int n = 0;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) n = 0;
  cache[dev] = n;
  return n;
}

}  // namespace pgb
