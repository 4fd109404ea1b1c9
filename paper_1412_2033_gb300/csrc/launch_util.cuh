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

// Kernels of the operator and of the iterations follow one another on a stream
// in hundreds, many of them a few microseconds long.  They are launched with
// programmatic stream serialisation: the next kernel's blocks are set up, and
// their prologue runs, as the blocks of the kernel before end.  Every thread of
// such a kernel calls grid_wait() before its first access to memory that a kernel
// writes: it returns when the grid before has completed and its writes are visible.
// Ahead of the wait it may only read what copies alone write, on the same stream and
// queued before the launch: the work items and plans of the batched launches (Arena,
// get_plan in batch.cu).  A copy is never a programmatic edge, so the first kernel
// behind it starts when it has completed and the later ones after that kernel, and
// the next copy to the same place waits for every kernel queued before it.
//
// Measured, the same kernels launched plainly and chained, one operator application
// among others: N = 63 FP32 31.2 -> 19.1 us (20.2 now; plain launches of the passes before
// the run-time plans 26.4), N = 2187 273 -> 262, N = 1023 79 -> 68, d = 3 N = 65 66 -> 53;
// FP64 N = 405 94 -> 83; bound pairs N = 2187 146 -> 141 ms, d = 3 N = 65 174 -> 140 ms.
// Where launches do not chain (ghb_profile records events between them) short passes
// take longer than those did.  Letting the next grid in
// earlier (griddepcontrol.launch_dependents after the wait) gives N = 63 18.6 us
// but N = 2187 310 us and its bound pair 164 ms: blocks that only wait hold shared
// memory and slots while the last blocks of the grid before still run.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// The pointer as read after the wait: no load through it, not even one the
// compiler takes for invariant (__restrict__), can be moved before the wait.
template <typename T>
__device__ __forceinline__ T* after_wait(T* p) {
  asm volatile("" : "+l"(p) : : "memory");
  return p;
}

template <typename... P, typename... A>
inline ghb_status launch_chained(void (*kernel)(P...), int64_t grid, int threads, size_t smem, cudaStream_t s,
                                 const A&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(grid));
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  GHB_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, args...));
  return GHB_OK;
}

// Index of the work item owning block `b` (items sorted by block_begin, n >= 1): a
// whole warp looks at 32 places a turn, so 1024 items take two loads one after the
// other instead of ten (256 solves of N = 31 .. 255: last axis 113 -> 110 us a
// launch, columns 45 -> 43 and 36 -> 34).  All lanes call it and get the index.
template <typename Item>
__device__ __forceinline__ int find_item(const Item* items, int n, int64_t b) {
  const int lane = threadIdx.x & 31;
  int lo = 0, len = n;
  while (len > 1) {
    const int step = (len + 31) / 32;
    const bool at = lane * step < len && items[lo + lane * step].block_begin <= b;
    const int k = 31 - __clz(__ballot_sync(0xffffffffu, at));   // lane 0 is always set
    lo += k * step;
    len = len - k * step < step ? len - k * step : step;
  }
  return lo;
}

}  // namespace ghb
