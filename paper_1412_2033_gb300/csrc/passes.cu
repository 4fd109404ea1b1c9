// Transform passes of the double-grid Ga operator (Algorithm 2 on the Fourier
// side, Cor. Ga_linsys; Lemma integ_eval_VM):
//
//   column pass  -- zero-pad Z_N -> Z_M and inverse DFT (or forward DFT and
//                   truncate Z_M -> Z_N) along one non-contiguous axis, for a
//                   tile of TW neighbouring lines held interleaved in shared
//                   memory (rows of TW contiguous entries are read and written);
//   row pass     -- the contiguous last axis, stored as a half spectrum:
//                   Hermitian completion, inverse DFT to real values, then
//                     MATVEC: multiply by A_M(x_m) and transform back,
//                     TOREAL: store the real values (the double-grid values
//                             A_M of eq. MBA_GA),
//                     ENERGY: accumulate the Gram sums
//                             (1/|M|) sum_m A_M(x_m) v_i(x_m).v_j(x_m).
//                   Two real lines share one complex transform (z = u + i v).
#include <algorithm>
#include <atomic>
#include <cmath>

#include "ghb_internal.cuh"
#include "passes_fx.cuh"
#include "passes_rt.cuh"

namespace ghb {

// Launchers defined by instantiation in the ct_*.cu units.
template <int M>
ghb_status launch_col_ct_m(int sign, int mode, const ColArgs& a, const CtTables& pl, cudaStream_t s);
template <int M>
ghb_status launch_row_ct_m(int NL, const RowArgs& a, const CtTables& pl, int rows_per_cta, cudaStream_t s);

ghb_status launch_col_ct(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s) {
  switch (pl.M) {
    case 162: return launch_col_ct_m<162>(sign, mode, a, pl.ct, s);
    case 486: return launch_col_ct_m<486>(sign, mode, a, pl.ct, s);
    case 1458: return launch_col_ct_m<1458>(sign, mode, a, pl.ct, s);
    case 4374: return launch_col_ct_m<4374>(sign, mode, a, pl.ct, s);
    case 2187: return launch_col_ct_m<2187>(sign, mode, a, pl.ct, s);
    case 72: return launch_col_ct_m<72>(sign, mode, a, pl.ct, s);
    case 135: return launch_col_ct_m<135>(sign, mode, a, pl.ct, s);
    case 270: return launch_col_ct_m<270>(sign, mode, a, pl.ct, s);
    default: break;
  }
  set_error("internal: no size-specialised kernels for M=" + std::to_string(pl.M));
  return GHB_ERR_INVALID;
}

ghb_status launch_row_ct(int NL, const RowArgs& a, const FftPlan& pl, int rows_per_cta, cudaStream_t s) {
  switch (pl.M) {
    case 162: return launch_row_ct_m<162>(NL, a, pl.ct, rows_per_cta, s);
    case 486: return launch_row_ct_m<486>(NL, a, pl.ct, rows_per_cta, s);
    case 1458: return launch_row_ct_m<1458>(NL, a, pl.ct, rows_per_cta, s);
    case 4374: return launch_row_ct_m<4374>(NL, a, pl.ct, rows_per_cta, s);
    case 2187: return launch_row_ct_m<2187>(NL, a, pl.ct, rows_per_cta, s);
    case 72: return launch_row_ct_m<72>(NL, a, pl.ct, rows_per_cta, s);
    case 135: return launch_row_ct_m<135>(NL, a, pl.ct, rows_per_cta, s);
    case 270: return launch_row_ct_m<270>(NL, a, pl.ct, rows_per_cta, s);
    default: break;
  }
  set_error("internal: no size-specialised kernels for M=" + std::to_string(pl.M));
  return GHB_ERR_INVALID;
}

// The size-specialised FP32 kernels run where they are compiled, the plan
// carries their input order and the autotuner chose them.
bool use_ct(const FftPlan& pl, bool tuned_on) { return pl.ct.perm != nullptr && ct_size(pl.M) && tuned_on; }

namespace {

int device_sms() {
  static std::atomic<int> cache{0};   // one device model per process
  int sms = cache.load(std::memory_order_relaxed);
  if (sms == 0) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
      sms = 152;
    cache.store(sms, std::memory_order_relaxed);
  }
  return sms;
}

}  // namespace

// FP64 columns per CTA: the widest tile (32-byte and longer row segments) that
// leaves room for three CTAs on an SM and makes at least two CTAs for each; an
// operand too small for that takes one column per CTA.
int fx_col_tile(int ls, int64_t columns) {
  for (int tw : {8, 4, 2}) {
    const size_t smem = static_cast<size_t>(tw) * ls * sizeof(fx2);
    if (smem <= 73 * 1024 && (columns + tw - 1) / tw >= 2 * device_sms()) return tw;
  }
  return 1;
}
// About one group of nine entries a thread and pass, whole warps.
int fx_threads(int M, int lines, int ls) {
  const size_t smem = static_cast<size_t>(lines) * ls * sizeof(fx2);
  const int full = smem > 110 * 1024 ? kFxThreads : (smem > 50 * 1024 ? kFxThreads / 2 : kFxThreads / 3);
  const int t = ((lines * M / 9 + 31) / 32) * 32;
  return t < 64 ? 64 : (t < full ? t : full);
}
// FP64 last-axis pass: the base group (one row, two where a row's real lines
// are odd in number), doubled while the threads it gives work to stay below a
// block of 256, the lines fit twice on an SM and two CTAs remain for each SM.
void fx_row_shape(int mode, int nfields, int ncomp, int M, int ls, int64_t rows, int* rows_per_cta, int* NL,
                  int* threads) {
  const int per_row = nfields * ncomp;
  int r = (mode != ROW_ENERGY && per_row % 2 == 1) ? 2 : 1;
  if (mode != ROW_ENERGY) {
    while (true) {
      const int nl = r * per_row;   // lines after doubling
      if (nl > kFxMaxLines || static_cast<size_t>(nl) * ls * sizeof(fx2) > 72 * 1024) break;
      if ((r * per_row / 2) * (M / 9) >= 256) break;
      if (rows / (2 * r) < 2 * device_sms()) break;
      r *= 2;
    }
  }
  *rows_per_cta = r;
  *NL = (r * per_row + 1) / 2;
  *threads = fx_threads(M, *NL, ls);
}

// FP32 run-time plans.  Columns per CTA: the widest tile (row segments of 8 TW
// bytes) that leaves room for three CTAs on an SM and makes two for each; four
// columns also as one CTA of 768 threads and from 1.6 CTAs for each SM (M = 2048,
// 1024 columns: 22 / 20 us with four, 28 / 23 with two; M = 1440, 702 columns: 21 /
// 18 with four, 19 / 14 with two).
int rt_col_tile(int M, int ls, int64_t columns) {
  for (int tw : {16, 8, 4}) {
    const size_t smem = static_cast<size_t>(tw) * ls * sizeof(float2);
    const int64_t ctas = (columns + tw - 1) / tw;
    if (smem <= (tw == 4 ? 150 : 73) * 1024 && 10 * ctas >= (tw == 4 ? 16 : 20) * device_sms()) return tw;
  }
  return 2 * column_stride(ls, 2, sizeof(float2)) * sizeof(float2) <= kPassSmem ? 2 : 1;
}
// More warps than the 24 that kernels of 80 registers keep on every SM.
bool rt_many_warps(int64_t blocks, int threads) {
  return blocks * (threads / 32) > int64_t(kRtThreads / 32) * device_sms();
}
// about one group of sixteen entries a thread and pass, whole warps
int rt_threads(int M, int lines, int ls) {
  const size_t smem = static_cast<size_t>(lines) * ls * sizeof(float2);
  const int full = smem > 110 * 1024 ? kRtThreads : (smem > 73 * 1024 ? kRtThreads / 2 : 256);
  const int t = ((lines * M / 16 + 31) / 32) * 32;
  return t < 64 ? 64 : (t < full ? t : full);
}
// Last axis: the least rows that fill complex lines (d = 2: one, d = 3: two rows,
// three lines), doubled while a block of 256 has threads without a group and two
// CTAs remain for each SM; `want` = 1 keeps the least, 2 doubles it once (d = 2:
// at every length whose two lines are admitted, as ghb_tune_set promises).
void rt_row_shape(int ncomp, int M, int ls, int64_t rows, int want, int* rows_per_cta, int* lines) {
  int r = ncomp == 2 ? 1 : 2, q = r * ncomp / 2;
  const size_t most = want == 2 && ncomp == 2 ? kPassSmem : 73 * 1024;
  while (want != 1 && 2 * q <= kRtMaxLines && static_cast<size_t>(2 * q) * ls * sizeof(float2) <= most &&
         (want == 2 || (q * (M / 16) < 192 && rows / (2 * r) >= 2 * device_sms()))) {
    r *= 2;
    q *= 2;
    if (want == 2) break;
  }
  *rows_per_cta = r;
  *lines = q;
}

template <>
ghb_status launch_col<double>(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s) {
  int TW = pl.tile[0];   // ghb_tune_set; 0 = by the operand
  if (TW <= 0) TW = fx_col_tile(pl.fx.ls, a.outer * a.inner);
  if (!col_admitted(pl.M, 1, sizeof(double2))) {
    set_error("transform length too large for one CTA: M=" + std::to_string(pl.M));
    return GHB_ERR_INVALID;
  }
  ColArgs b = a;
  if (mode != COL_PUPDATE) b.pold = nullptr;
  return launch_fx_col(sign, b, pl.fx, TW, s);
}

template <>
ghb_status launch_col<float>(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s) {
  if (use_ct(pl, pl.ct_col != 0)) return launch_col_ct(sign, mode, a, pl, s);
  // the kernel's 32-bit offsets are row i times `inner` inside one outer index (RtColIn)
  if (std::max<int64_t>(std::max(a.Lin, a.Lout), pl.M) * a.inner >= (int64_t(1) << 31)) {
    set_error("column pass with 2^31 entries or more in one outer index");
    return GHB_ERR_INVALID;
  }
  int TW = pl.tile[1];   // ghb_tune_set; 0 = by the operand
  if (TW <= 0) TW = rt_col_tile(pl.M, pl.rt.ls, a.outer * a.inner);
  if (!col_admitted(pl.M, 1, sizeof(float2))) {
    set_error("transform length too large for one CTA: M=" + std::to_string(pl.M));
    return GHB_ERR_INVALID;
  }
  ColArgs b = a;
  if (mode != COL_PUPDATE) b.pold = nullptr;
  return launch_rt_col(sign, b, pl.rt, TW, s);
}

// Rows a CTA transforms together in the operator's last-axis pass (d = 2:
// 1 or 2, the tuned value or by size: two rows for M <= 2048, one above; odd
// line counts always pair two rows).
void row_lines(int mode, int nfields, int ncomp, int M, int rows32, int* rows_per_cta, int* NL) {
  const int per_row = nfields * ncomp;
  int r = 1;
  if (mode == ROW_MATVEC || mode == ROW_TOREAL) r = (per_row % 2 == 1) ? 2 : 1;
  if (mode == ROW_MATVEC && per_row == 2) r = (rows32 == 1 || rows32 == 2) ? rows32 : (M <= 2048 ? 2 : 1);
  *rows_per_cta = r;
  *NL = (r * per_row + 1) / 2;
}

template <>
ghb_status launch_col_batch<float>(int sign, int mode, const ColItem* items, int n, int64_t blocks, size_t smem,
                                   int threads, cudaStream_t s) {
  return launch_rt_col_batch(sign, mode == COL_PUPDATE, items, n, blocks, smem, threads, s);
}
template <>
ghb_status launch_col_batch<double>(int sign, int, const ColItem* items, int n, int64_t blocks, size_t smem, int threads,
                                    cudaStream_t s) {
  return launch_fx_col_batch(sign, items, n, blocks, smem, threads, s);
}

template <>
ghb_status launch_row_batch<float>(int mode, const RowItem* items, int n, int64_t blocks, size_t smem, int threads,
                                   cudaStream_t s) {
  if (mode == ROW_MATVEC) return launch_rt_row_batch(items, n, blocks, smem, threads, s);
  set_error("internal: unsupported batched row pass");
  return GHB_ERR_INVALID;
}
template <>
ghb_status launch_row_batch<double>(int mode, const RowItem* items, int n, int64_t blocks, size_t smem, int threads,
                                    cudaStream_t s) {
  return launch_fx_row_batch(mode, items, n, blocks, smem, threads, s);
}

template <>
ghb_status launch_row<float>(int mode, const RowArgs& a, const FftPlan& pl, cudaStream_t s) {
  int rows_per_cta = 1, NL = 1;
  row_lines(mode, a.nfields, a.ncomp, pl.M, pl.rows32, &rows_per_cta, &NL);
  if (mode == ROW_MATVEC) {   // set-up and Gram passes run in FP64 only
    if (use_ct(pl, (a.ncomp == 3 ? pl.ct_row3 : pl.ct_row) != 0)) return launch_row_ct(NL, a, pl, rows_per_cta, s);
    if (!row_admitted(pl.M, NL, sizeof(float2))) {
      set_error("row transform too large for one CTA: M=" + std::to_string(pl.M));
      return GHB_ERR_INVALID;
    }
    int lines = 1;
    rt_row_shape(a.ncomp, pl.M, pl.rt.ls, a.rows, pl.rows32, &rows_per_cta, &lines);
    return launch_rt_row(a, pl.rt, rows_per_cta, lines, s);
  }
  set_error("internal: unsupported FP32 row pass");
  return GHB_ERR_INVALID;
}

template <>
ghb_status launch_row<double>(int mode, const RowArgs& a, const FftPlan& pl, cudaStream_t s) {
  int rows_per_cta = 1, NL = 1, threads = 256;
  row_lines(mode, a.nfields, a.ncomp, pl.M, 0, &rows_per_cta, &NL);
  if (!row_admitted(pl.M, NL, sizeof(double2))) {
    set_error("row transform too large for one CTA: M=" + std::to_string(pl.M));
    return GHB_ERR_INVALID;
  }
  fx_row_shape(mode, a.nfields, a.ncomp, pl.M, pl.fx.ls, a.rows, &rows_per_cta, &NL, &threads);
  return launch_fx_row(mode, a, pl.fx, rows_per_cta, NL, threads, s);
}

}  // namespace ghb
