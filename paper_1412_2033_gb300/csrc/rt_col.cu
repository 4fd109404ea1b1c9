// Column-pass kernels of the FP32 run-time plans; see passes_rt.cuh.
#include "launch_util.cuh"
#include "passes_rt.cuh"

namespace ghb {

template <int SIGN, bool UPDATE>
__global__ void __launch_bounds__(kRtThreads, 1)
    rt_col_kernel(const __grid_constant__ ColArgs a, const __grid_constant__ FxPlan f, int TW) {
  rt_col_body<SIGN, UPDATE>(a, f, TW, blockIdx.x);
}

template <int SIGN, bool UPDATE, int THREADS>
__global__ void __launch_bounds__(THREADS, 1) rt_col_kernel_batch(const ColItem* __restrict__ items, int n) {
  __shared__ int s_item;
  if (threadIdx.x < 32) s_item = find_item(items, n, blockIdx.x);
  __syncthreads();
  const ColItem& it = items[s_item];
  rt_col_body<SIGN, UPDATE>(it.a, it.pl->rt, it.tile, blockIdx.x - it.block_begin);
}

namespace {

template <int SIGN, bool UPDATE>
ghb_status col_launch(const ColArgs& a, const FxPlan& f, int TW, cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(rt_col_kernel<SIGN, UPDATE>, kPassSmem, mask));
  const size_t smem = static_cast<size_t>(TW) * column_stride(f.ls, TW, sizeof(float2)) * sizeof(float2);
  const int64_t grid = (a.outer * a.inner + TW - 1) / TW;
  return launch_chained(rt_col_kernel<SIGN, UPDATE>, grid, rt_threads(f.M, TW, f.ls), smem, s, a, f, TW);
}

template <int SIGN, bool UPDATE, int THREADS>
ghb_status col_launch_batch_of(const ColItem* items, int n, int64_t blocks, size_t smem, int threads, cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(rt_col_kernel_batch<SIGN, UPDATE, THREADS>, kPassSmem, mask));
  return launch_chained(rt_col_kernel_batch<SIGN, UPDATE, THREADS>, blocks, threads, smem, s, items, n);
}
template <int SIGN, bool UPDATE>
ghb_status col_launch_batch(const ColItem* items, int n, int64_t blocks, size_t smem, int threads, cudaStream_t s) {
  if (rt_many_warps(blocks, threads))
    return col_launch_batch_of<SIGN, UPDATE, kRtManyThreads>(items, n, blocks, smem, threads, s);
  return col_launch_batch_of<SIGN, UPDATE, kRtThreads>(items, n, blocks, smem, threads, s);
}

}  // namespace

ghb_status launch_rt_col(int sign, const ColArgs& a, const FxPlan& f, int TW, cudaStream_t s) {
  if (sign < 0) return col_launch<-1, false>(a, f, TW, s);
  return a.pold != nullptr ? col_launch<+1, true>(a, f, TW, s) : col_launch<+1, false>(a, f, TW, s);
}

ghb_status launch_rt_col_batch(int sign, bool update, const ColItem* items, int n, int64_t blocks, size_t smem,
                               int threads, cudaStream_t s) {
  if (sign < 0) return col_launch_batch<-1, false>(items, n, blocks, smem, threads, s);
  return update ? col_launch_batch<+1, true>(items, n, blocks, smem, threads, s)
                : col_launch_batch<+1, false>(items, n, blocks, smem, threads, s);
}

}  // namespace ghb
