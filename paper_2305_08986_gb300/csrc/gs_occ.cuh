// Device properties the launchers size their grids by (cached per device).
#pragma once
#include "gs_batch.cuh"

namespace gs {

inline int device_index() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}

inline int sm_count() {
  static std::atomic<int> cache[kMaxDevices];
  const int dev = device_index();
  if (dev >= 0 && cache[dev].load(std::memory_order_relaxed) > 0) return cache[dev].load(std::memory_order_relaxed);
  int v = 0;
  if (cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev < 0 ? 0 : dev) != cudaSuccess || v <= 0) v = 1;
  if (dev >= 0) cache[dev].store(v, std::memory_order_relaxed);
  return v;
}

// Resident CTAs per SM of the kernel with `smem` bytes of dynamic shared memory (per device; one
// shared-memory size per kernel).
template <class K>
int ctas_per_sm(size_t smem) {
  static std::atomic<size_t> enabled[kMaxDevices];
  static std::atomic<int> cache[kMaxDevices];
  const int dev = device_index();
  if (dev >= 0 && cache[dev].load(std::memory_order_relaxed) > 0) return cache[dev].load(std::memory_order_relaxed);
  int n = 1;
  if (ensure_dynamic_smem(k_one<K>, smem, enabled) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_one<K>, K::THREADS, smem) == cudaSuccess && n > 0) {
    if (dev >= 0) cache[dev].store(n, std::memory_order_relaxed);
  } else {
    cudaGetLastError();
    n = 1;
  }
  return n;
}

}  // namespace gs
