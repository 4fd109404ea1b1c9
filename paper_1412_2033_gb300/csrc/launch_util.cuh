// Launch helpers shared by the transform-pass units.
#pragma once

#include <atomic>

#include "ghb_internal.cuh"

namespace ghb {

// The dynamic shared-memory limit of kernel `func` raised to `bytes` on the
// current device.  The attribute belongs to the device's context, so it is set
// once per device (bit `dev` of `mask`, one mask per kernel); two host threads
// may both set it, which is harmless.  Devices beyond 63 set it every time.
template <typename F>
inline ghb_status ensure_dyn_smem(F* func, int bytes, std::atomic<unsigned long long>& mask) {
  int dev = 0;
  GHB_CUDA_TRY(cudaGetDevice(&dev));
  const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;
  if (bit == 0 || !(mask.load(std::memory_order_acquire) & bit)) {
    GHB_CUDA_TRY(cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    mask.fetch_or(bit, std::memory_order_release);
  }
  return GHB_OK;
}

// Index of the work item owning block `b` (items sorted by block_begin).
template <typename Item>
__device__ __forceinline__ int find_item(const Item* items, int n, int64_t b) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (items[mid].block_begin <= b) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

}  // namespace ghb
