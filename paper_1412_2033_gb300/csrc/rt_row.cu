// Last-axis kernels of the FP32 run-time plans; see passes_rt.cuh.
#include "launch_util.cuh"
#include "passes_rt.cuh"

namespace ghb {

template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1)
    rt_row_kernel(const __grid_constant__ RowArgs a, const __grid_constant__ FxPlan f, int rows_per_cta, int lines) {
  rt_row_body(a, f, rows_per_cta, lines, blockIdx.x, gridDim.x);
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1) rt_row_kernel_batch(const RowItem* __restrict__ items, int n) {
  __shared__ int s_item;
  if (threadIdx.x < 32) s_item = find_item(items, n, blockIdx.x);
  __syncthreads();
  const RowItem& it = items[s_item];
  rt_row_body(it.a, it.pl->rt, it.rows_per_cta, it.lines, blockIdx.x - it.block_begin, it.nblocks);
}

namespace {

template <int THREADS>
ghb_status row_launch(const RowArgs& a, const FxPlan& f, int64_t grid, int threads, int rows_per_cta, int lines,
                      cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(rt_row_kernel<THREADS>, kPassSmem, mask));
  const size_t smem = static_cast<size_t>(lines) * f.ls * sizeof(float2);
  return launch_chained(rt_row_kernel<THREADS>, grid, threads, smem, s, a, f, rows_per_cta, lines);
}

template <int THREADS>
ghb_status row_launch_batch(const RowItem* items, int n, int64_t blocks, size_t smem, int threads, cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(rt_row_kernel_batch<THREADS>, kPassSmem, mask));
  return launch_chained(rt_row_kernel_batch<THREADS>, blocks, threads, smem, s, items, n);
}

}  // namespace

ghb_status launch_rt_row(const RowArgs& a, const FxPlan& f, int rows_per_cta, int lines, cudaStream_t s) {
  const int64_t grid = (a.rows + rows_per_cta - 1) / rows_per_cta;
  const int threads = rt_threads(f.M, lines, f.ls);
  if (rt_many_warps(grid, threads)) return row_launch<kRtManyThreads>(a, f, grid, threads, rows_per_cta, lines, s);
  return row_launch<kRtThreads>(a, f, grid, threads, rows_per_cta, lines, s);
}

ghb_status launch_rt_row_batch(const RowItem* items, int n, int64_t blocks, size_t smem, int threads, cudaStream_t s) {
  if (rt_many_warps(blocks, threads)) return row_launch_batch<kRtManyThreads>(items, n, blocks, smem, threads, s);
  return row_launch_batch<kRtThreads>(items, n, blocks, smem, threads, s);
}

}  // namespace ghb
