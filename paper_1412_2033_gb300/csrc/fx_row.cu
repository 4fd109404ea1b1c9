// Last-axis kernels of the FP64 (fixed-point) transforms; see passes_fx.cuh.
#include "launch_util.cuh"
#include "passes_fx.cuh"

namespace ghb {

template <int MODE>
__global__ void __launch_bounds__(kFxThreads, kFxBlocks)
    fx_row_kernel(const __grid_constant__ RowArgs a, const __grid_constant__ FxPlan f, int rows_per_cta, int NL) {
  fx_row_body<MODE>(a, f, rows_per_cta, NL, blockIdx.x, gridDim.x);
}

template <int MODE>
__global__ void __launch_bounds__(kFxThreads, kFxBlocks) fx_row_kernel_batch(const RowItem* __restrict__ items, int n) {
  __shared__ int s_item;
  if (threadIdx.x < 32) s_item = find_item(items, n, blockIdx.x);
  __syncthreads();
  const RowItem& it = items[s_item];
  fx_row_body<MODE>(it.a, it.pl->fx, it.rows_per_cta, it.lines, blockIdx.x - it.block_begin, it.nblocks);
}

namespace {

template <int MODE>
ghb_status row_launch(const RowArgs& a, const FxPlan& f, int rows_per_cta, int NL, int threads, cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(fx_row_kernel<MODE>, kPassSmem, mask));
  const size_t smem = static_cast<size_t>(NL) * f.ls * sizeof(fx2);
  int64_t grid = (a.rows + rows_per_cta - 1) / rows_per_cta;
  if (MODE == ROW_ENERGY && grid > 1024) grid = 1024;   // partials hold 1024 x 6 doubles
  return launch_chained(fx_row_kernel<MODE>, grid, threads, smem, s, a, f, rows_per_cta, NL);
}

template <int MODE>
ghb_status row_launch_batch(const RowItem* items, int n, int64_t blocks, size_t smem, int threads,
                            cudaStream_t s) {
  static std::atomic<unsigned long long> mask{0};
  TRY_STATUS(ensure_dyn_smem(fx_row_kernel_batch<MODE>, kPassSmem, mask));
  return launch_chained(fx_row_kernel_batch<MODE>, blocks, threads, smem, s, items, n);
}

}  // namespace

ghb_status launch_fx_row(int mode, const RowArgs& a, const FxPlan& f, int rows_per_cta, int NL, int threads,
                         cudaStream_t s) {
  switch (mode) {
    case ROW_MATVEC: return row_launch<ROW_MATVEC>(a, f, rows_per_cta, NL, threads, s);
    case ROW_TOREAL: return row_launch<ROW_TOREAL>(a, f, rows_per_cta, NL, threads, s);
    default: return row_launch<ROW_ENERGY>(a, f, rows_per_cta, NL, threads, s);
  }
}

ghb_status launch_fx_row_batch(int mode, const RowItem* items, int n, int64_t blocks, size_t smem, int threads,
                               cudaStream_t s) {
  switch (mode) {
    case ROW_MATVEC: return row_launch_batch<ROW_MATVEC>(items, n, blocks, smem, threads, s);
    case ROW_ENERGY: return row_launch_batch<ROW_ENERGY>(items, n, blocks, smem, threads, s);
    default: break;
  }
  set_error("internal: unsupported batched row pass");
  return GHB_ERR_INVALID;
}

}  // namespace ghb
