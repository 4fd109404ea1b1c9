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

namespace ghb {

// Launchers defined by instantiation in the col_*.cu / row_*.cu units.
template <typename T, int TW, int MCT = 0>
ghb_status launch_col_tw(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s);
template <typename T, int NL, int MODE>
ghb_status launch_row_nl(const RowArgs& a, const FftPlan& pl, int rows_per_cta, cudaStream_t s);
template <typename T, int TW>
ghb_status launch_col_batch_tw(int sign, int mode, const ColItem* items, int n, int64_t blocks, size_t smem, int threads,
                               cudaStream_t s);
template <typename T, int NL, int MODE>
ghb_status launch_row_batch_nl(const RowItem* items, int n, int64_t blocks, size_t smem, int threads, cudaStream_t s);

template <typename T, int M>
ghb_status launch_col_ct_m(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s);
template <typename T, int M>
ghb_status launch_row_ct_m(int NL, const RowArgs& a, const FftPlan& pl, int rows_per_cta, cudaStream_t s);

template <typename T>
ghb_status launch_col_ct(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s) {
  switch (pl.M) {
    case 162: return launch_col_ct_m<T, 162>(sign, mode, a, pl, s);
    case 486: return launch_col_ct_m<T, 486>(sign, mode, a, pl, s);
    case 1458: return launch_col_ct_m<T, 1458>(sign, mode, a, pl, s);
    case 4374: return launch_col_ct_m<T, 4374>(sign, mode, a, pl, s);
    case 2187: return launch_col_ct_m<T, 2187>(sign, mode, a, pl, s);
    case 72: return launch_col_ct_m<T, 72>(sign, mode, a, pl, s);
    case 135: return launch_col_ct_m<T, 135>(sign, mode, a, pl, s);
    case 270: return launch_col_ct_m<T, 270>(sign, mode, a, pl, s);
    default: break;
  }
  set_error("internal: no size-specialised kernels for M=" + std::to_string(pl.M));
  return GHB_ERR_INVALID;
}
template ghb_status launch_col_ct<float>(int, int, const ColArgs&, const FftPlan&, cudaStream_t);

template <typename T>
ghb_status launch_row_ct(int NL, const RowArgs& a, const FftPlan& pl, int rows_per_cta, cudaStream_t s) {
  switch (pl.M) {
    case 162: return launch_row_ct_m<T, 162>(NL, a, pl, rows_per_cta, s);
    case 486: return launch_row_ct_m<T, 486>(NL, a, pl, rows_per_cta, s);
    case 1458: return launch_row_ct_m<T, 1458>(NL, a, pl, rows_per_cta, s);
    case 4374: return launch_row_ct_m<T, 4374>(NL, a, pl, rows_per_cta, s);
    case 2187: return launch_row_ct_m<T, 2187>(NL, a, pl, rows_per_cta, s);
    case 72: return launch_row_ct_m<T, 72>(NL, a, pl, rows_per_cta, s);
    case 135: return launch_row_ct_m<T, 135>(NL, a, pl, rows_per_cta, s);
    case 270: return launch_row_ct_m<T, 270>(NL, a, pl, rows_per_cta, s);
    default: break;
  }
  set_error("internal: no size-specialised kernels for M=" + std::to_string(pl.M));
  return GHB_ERR_INVALID;
}
template ghb_status launch_row_ct<float>(int, const RowArgs&, const FftPlan&, int, cudaStream_t);

// The size-specialised FP32 kernels run where they are compiled, the plan
// carries their input order and the autotuner chose them.
bool use_ct(const FftPlan& pl, bool tuned_on) { return pl.perm_ct != nullptr && ct_size(pl.M) && tuned_on; }

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

// Columns per CTA of a runtime-plan column pass over `outer` x `inner` lines:
// the widest tile (coalesced rows of up to 16 entries) whose CTAs still fill
// the device three times over; operands too narrow for that take the tile
// with the most CTAs.  Wide operands (the axis-1 pass in 3-D) get wide tiles,
// narrow ones (2-D operands of small N) narrow ones.
int auto_tile(int M, int64_t outer, int64_t inner, int elem_bytes) {
  const int sms = device_sms();
  int fallback = 0;
  for (int tw : {16, 8, 4, 2, 1}) {
    const size_t smem = col_smem_bytes(M, tw, elem_bytes);
    if (smem > 220 * 1024) continue;
    const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(4, (227 * 1024) / static_cast<int64_t>(smem)));
    const int64_t ctas = outer * ((inner + tw - 1) / tw);
    if (ctas >= 3 * per_sm * sms) return tw;
    fallback = tw;   // the narrowest fitting tile: the most CTAs
  }
  return fallback > 0 ? fallback : 1;
}

// FP64 columns per CTA: the widest tile (32-byte and longer row segments) that
// leaves room for three CTAs on an SM and makes at least two CTAs for each; an
// operand too small for that takes one column per CTA.
int fx_col_tile(const FftPlan& pl, int64_t columns) {
  for (int tw : {8, 4, 2}) {
    const size_t smem = static_cast<size_t>(tw) * pl.fx.ls * sizeof(fx2);
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

template <>
ghb_status launch_col<double>(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s) {
  int TW = pl.tile[0];   // ghb_tune_set; 0 = by the operand
  if (TW <= 0 || static_cast<size_t>(TW) * pl.fx.ls * sizeof(fx2) > 220 * 1024)
    TW = fx_col_tile(pl, a.outer * a.inner);
  if (col_smem_bytes(pl.M, 1, sizeof(double2)) > 220 * 1024) {
    set_error("transform length too large for one CTA: M=" + std::to_string(pl.M));
    return GHB_ERR_INVALID;
  }
  ColArgs b = a;
  if (mode != COL_PUPDATE) b.pold = nullptr;
  return launch_fx_col(sign, b, pl, TW, s);
}

template <>
ghb_status launch_col<float>(int sign, int mode, const ColArgs& a, const FftPlan& pl, cudaStream_t s) {
  using T = float;
  using C = float2;
  if (use_ct(pl, pl.ct_col != 0)) return launch_col_ct<T>(sign, mode, a, pl, s);
  const int forced = pl.tile[1];   // ghb_tune_set; 0 = by the operand
  const int TW = forced > 0 ? forced : auto_tile(pl.M, a.outer, a.inner, sizeof(C));
  if (col_smem_bytes(pl.M, TW, sizeof(C)) > 220 * 1024) {
    set_error("transform length too large for one CTA: M=" + std::to_string(pl.M));
    return GHB_ERR_INVALID;
  }
  switch (TW) {
    case 1: return launch_col_tw<T, 1>(sign, mode, a, pl, s);
    case 2: return launch_col_tw<T, 2>(sign, mode, a, pl, s);
    case 4: return launch_col_tw<T, 4>(sign, mode, a, pl, s);
    case 8: return launch_col_tw<T, 8>(sign, mode, a, pl, s);
    case 16: return launch_col_tw<T, 16>(sign, mode, a, pl, s);
    default: break;
  }
  set_error("internal: bad tile width");
  return GHB_ERR_INVALID;
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
ghb_status launch_col_batch<float>(int sign, int mode, int TW, const ColItem* items, int n, int64_t blocks,
                                   size_t smem, int threads, cudaStream_t s) {
  using T = float;
  switch (TW) {
    case 1: return launch_col_batch_tw<T, 1>(sign, mode, items, n, blocks, smem, threads, s);
    case 2: return launch_col_batch_tw<T, 2>(sign, mode, items, n, blocks, smem, threads, s);
    case 4: return launch_col_batch_tw<T, 4>(sign, mode, items, n, blocks, smem, threads, s);
    case 8: return launch_col_batch_tw<T, 8>(sign, mode, items, n, blocks, smem, threads, s);
    case 16: return launch_col_batch_tw<T, 16>(sign, mode, items, n, blocks, smem, threads, s);
    default: break;
  }
  set_error("internal: bad tile width");
  return GHB_ERR_INVALID;
}
template <>
ghb_status launch_col_batch<double>(int sign, int, int TW, const ColItem* items, int n, int64_t blocks, size_t smem,
                                    int threads, cudaStream_t s) {
  return launch_fx_col_batch(sign, TW, items, n, blocks, smem, threads, s);
}

template <>
ghb_status launch_row_batch<float>(int mode, int NL, const RowItem* items, int n, int64_t blocks, size_t smem,
                                   int threads, cudaStream_t s) {
  using T = float;
  if (mode == ROW_MATVEC) {
    if (NL == 1) return launch_row_batch_nl<T, 1, ROW_MATVEC>(items, n, blocks, smem, threads, s);
    if (NL == 2) return launch_row_batch_nl<T, 2, ROW_MATVEC>(items, n, blocks, smem, threads, s);
    if (NL == 3) return launch_row_batch_nl<T, 3, ROW_MATVEC>(items, n, blocks, smem, threads, s);
  }
  set_error("internal: unsupported batched row pass");
  return GHB_ERR_INVALID;
}
template <>
ghb_status launch_row_batch<double>(int mode, int NL, const RowItem* items, int n, int64_t blocks, size_t smem,
                                    int threads, cudaStream_t s) {
  return launch_fx_row_batch(mode, NL, items, n, blocks, smem, threads, s);
}

template <>
ghb_status launch_row<float>(int mode, const RowArgs& a, const FftPlan& pl, cudaStream_t s) {
  using T = float;
  int rows_per_cta = 1, NL = 1;
  row_lines(mode, a.nfields, a.ncomp, pl.M, pl.rows32, &rows_per_cta, &NL);
  if (mode == ROW_MATVEC) {   // set-up and Gram passes run in FP64 only
    if (use_ct(pl, pl.ct_row != 0)) return launch_row_ct<T>(NL, a, pl, rows_per_cta, s);
    switch (NL) {
      case 1: return launch_row_nl<T, 1, ROW_MATVEC>(a, pl, rows_per_cta, s);
      case 2: return launch_row_nl<T, 2, ROW_MATVEC>(a, pl, rows_per_cta, s);
      case 3: return launch_row_nl<T, 3, ROW_MATVEC>(a, pl, rows_per_cta, s);
      default: break;
    }
  }
  set_error("internal: unsupported row-pass line count");
  return GHB_ERR_INVALID;
}

template <>
ghb_status launch_row<double>(int mode, const RowArgs& a, const FftPlan& pl, cudaStream_t s) {
  int rows_per_cta = 1, NL = 1, threads = 256;
  row_lines(mode, a.nfields, a.ncomp, pl.M, 0, &rows_per_cta, &NL);
  if (padded_elems<double2>(static_cast<size_t>(pl.M) * NL) * sizeof(double2) > 200 * 1024) {
    set_error("row transform too large for one CTA: M=" + std::to_string(pl.M));
    return GHB_ERR_INVALID;
  }
  fx_row_shape(mode, a.nfields, a.ncomp, pl.M, pl.fx.ls, a.rows, &rows_per_cta, &NL, &threads);
  return launch_fx_row(mode, a, pl, rows_per_cta, NL, threads, s);
}

}  // namespace ghb
