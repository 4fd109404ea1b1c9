// Column-pass kernels of the FP64 (fixed-point) transforms; see passes_fx.cuh.
#include "launch_util.cuh"
#include "passes_fx.cuh"

namespace ghb {

template <int SIGN>
__global__ void __launch_bounds__(kFxThreads, kFxBlocks)
    fx_col_kernel(const __grid_constant__ ColArgs a, const __grid_constant__ FxPlan f, int TW) {
  fx_col_body<SIGN>(a, f, TW, blockIdx.x);
}

template <int SIGN>
__global__ void __launch_bounds__(kFxThreads, kFxBlocks) fx_col_kernel_batch(const ColItem* __restrict__ items, int n) {
  __shared__ int s_item;
  if (threadIdx.x < 32) s_item = find_item(items, n, blockIdx.x);
  __syncthreads();
  const ColItem& it = items[s_item];
  fx_col_body<SIGN>(it.a, it.pl->fx, it.tile, blockIdx.x - it.block_begin);
}

namespace {

template <int SIGN>
ghb_status col_launch(const ColArgs& a, const FxPlan& f, int TW, cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(fx_col_kernel<SIGN>, kPassSmem, mask));
  const size_t smem = static_cast<size_t>(TW) * column_stride(f.ls, TW, sizeof(fx2)) * sizeof(fx2);
  const int64_t grid = (a.outer * a.inner + TW - 1) / TW;
  return launch_chained(fx_col_kernel<SIGN>, grid, fx_threads(f.M, TW, f.ls), smem, s, a, f, TW);
}

template <int SIGN>
ghb_status col_launch_batch(const ColItem* items, int n, int64_t blocks, size_t smem, int threads,
                            cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(fx_col_kernel_batch<SIGN>, kPassSmem, mask));
  return launch_chained(fx_col_kernel_batch<SIGN>, blocks, threads, smem, s, items, n);
}

}  // namespace

ghb_status launch_fx_col(int sign, const ColArgs& a, const FxPlan& f, int TW, cudaStream_t s) {
  return sign > 0 ? col_launch<+1>(a, f, TW, s) : col_launch<-1>(a, f, TW, s);
}

ghb_status launch_fx_col_batch(int sign, const ColItem* items, int n, int64_t blocks, size_t smem, int threads,
                               cudaStream_t s) {
  return sign > 0 ? col_launch_batch<+1>(items, n, blocks, smem, threads, s)
                  : col_launch_batch<-1>(items, n, blocks, smem, threads, s);
}

}  // namespace ghb
