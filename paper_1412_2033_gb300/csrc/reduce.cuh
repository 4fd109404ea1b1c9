// Deterministic block reductions (fixed shuffle tree, fixed block order).
#pragma once

#include <cuda_runtime.h>

namespace ghb {

// A thread's part of an inner product: a plain sum in the field's precision or, in the
// batched kernels on FP32 fields (PAIR), one entry's products in FP32 and the entries in
// two floats with the rounding of every sum kept (Knuth's two-sum), so that a thread
// may take several entries where it took one and its sum is no coarser.  An entry
// starts from open() and ends in close().
template <typename T, bool PAIR>
struct ThreadSum {
  T v = T(0);
  __host__ __device__ __forceinline__ T open() const { return v; }
  __host__ __device__ __forceinline__ void close(T s) { v = s; }
  __host__ __device__ __forceinline__ double total() const { return v; }
};
template <>
struct ThreadSum<float, true> {
  float v = 0.0f, low = 0.0f;
  __host__ __device__ __forceinline__ float open() const { return 0.0f; }
  __host__ __device__ __forceinline__ void close(float s) {
    const float t = v + s, u = t - v;
    low += (v - (t - u)) + (s - u);
    v = t;
  }
  __host__ __device__ __forceinline__ double total() const { return static_cast<double>(v) + static_cast<double>(low); }
};

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum of one double per thread; the result is valid in thread 0.  `scratch`
// holds 32 doubles of shared memory.  Contains barriers: call from all threads.
__device__ __forceinline__ double block_sum(double v, double* scratch) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) scratch[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    r = (lane < nw) ? scratch[lane] : 0.0;
    r = warp_sum(r);
  }
  return r;
}

// The same for blocks of at most 256 threads with scratch for 256 doubles: one
// warp adds eight values a lane before the tree, 12 FP64 instructions instead of
// 45 on a pipe that takes one warp's in 16 cycles (bound pairs: d = 3 N = 65 140.7 ->
// 136.3 ms, d = 2 N = 511 21.6 -> 20.6, 64 mixed microstructures 239.5 -> 236.7).
__device__ __forceinline__ double block_sum_wide(double v, double* scratch) {
  __syncthreads();
  scratch[threadIdx.x] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x < 32) {
    r = scratch[threadIdx.x];
#pragma unroll
    for (int i = 1; i < 8; ++i)
      if (threadIdx.x + 32 * i < blockDim.x) r += scratch[threadIdx.x + 32 * i];
    r = warp_sum(r);
  }
  return r;
}

}  // namespace ghb
