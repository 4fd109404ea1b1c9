// Kernel templates of the size-specialised FP32 transform passes (fft_ct.cuh) of
// the double-grid Ga operator (Algorithm 2 on the Fourier side, Cor. Ga_linsys;
// Lemma integ_eval_VM):
//
//   column pass  -- zero-pad Z_N -> Z_M and inverse DFT (or forward DFT and
//                   truncate Z_M -> Z_N) along one non-contiguous axis, for a
//                   tile of TW neighbouring lines held interleaved in shared
//                   memory (rows of TW contiguous entries are read and written);
//   row pass     -- the contiguous last axis, stored as a half spectrum:
//                   Hermitian completion, inverse DFT to real values, multiply
//                   by A_M(x_m) and transform back.  Two real lines share one
//                   complex transform (z = u + i v).
//
// Every other length, and FP64, runs passes_rt.cuh and passes_fx.cuh.  The
// templates are instantiated in one translation unit per length.
#pragma once

#include <algorithm>
#include <atomic>
#include <cmath>
#include <mutex>

#include "fft_ct.cuh"
#include "ghb_internal.cuh"
#include "launch_util.cuh"
#include "reduce.cuh"

namespace ghb {

// ---------------------------------------------------------------------------
// asynchronous global -> shared copies (cp.async): every thread issues its
// copies back to back and waits once, so a CTA's loads are all in flight
// together instead of one dependent load per loop iteration.
// ---------------------------------------------------------------------------
template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst_smem, const void* src) {
  const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst_smem));
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
// wait until at most N of this thread's committed groups are still in flight
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }

// Butterflies of one line in the pass with the fewest (the size-specialised
// plan of length M): a CTA of the last-axis pass keeps all its threads busy
// only if its interleaved lines times this count reach its thread count.
template <int M>
__host__ __device__ constexpr int ct_min_units() {
  constexpr CtPlan P = ct_plan(M);
  int mn = M;
  for (int i = 0; i < P.npass; ++i) {
    const int u = M / (P.ra[i] * P.rb[i] * P.rc[i]);
    if (u < mn) mn = u;
  }
  return mn;
}
// Threads of a column-pass CTA: one thread per butterfly of the pass with the
// fewest (TW lines of ct_min_units each), in whole warps, between 128 and 672.
// At M = 4374 the 4 x 162 radix-27 butterflies of a tile take one round of 672
// threads instead of two rounds of 512, the second about a quarter full: axis-1
// inverse 68 -> 60 us, forward 64 -> 61 us.  672 threads leave 80 registers,
// which the inverse pass with the p update exceeds (it spilled and measured 89
// against 86 us), so the p-update variants keep 512.  col_min_blocks keeps the
// register budget of a full block.
template <int TW, int MCT, int MODE>
__host__ __device__ constexpr int col_threads() {
  constexpr int full = MODE == COL_PUPDATE ? 512 : 672;
  int t = ((ct_min_units<MCT>() * TW + 31) / 32) * 32;
  if (t < 128) t = 128;
  return t < full ? t : full;
}
// Resident blocks the compiler must allow for: as many as make up a full
// block's threads; one fewer when that leaves fewer than the 96 registers a
// radix-27 group needs (448 threads at M = 1458 were held to 72 registers by two
// blocks and spilled 208 bytes: p-update inverse pass 19.4 -> 17.0 us).
template <int TW, int MCT, int MODE>
__host__ __device__ constexpr int col_min_blocks() {
  constexpr int t = col_threads<TW, MCT, MODE>();
  int b = (512 + t - 1) / t;
  if (b > 1 && 65536 / (b * t) < 96) --b;
  return b;
}

// ---------------------------------------------------------------------------
// column pass: block `bid` of one operand handles tile (o, j0..j0+TW)
// ---------------------------------------------------------------------------
// Input of the size-specialised inverse column transform: entry n of tile
// line t is input row i(n) = n + half (n <= half) or n - M + half
// (n >= M - half), zero in between; with UPDATE the entry is r + beta p_old
// and is written back to p_new once all of a unit's entries are loaded.
// off[t] is the element offset of row 0 of line t's column (a tile's lines
// may belong to different outer indices); offsets are 32-bit (the launcher
// rejects operands of 2^31 entries or more), which keeps a unit's indices in
// one register each until the write-back.
template <typename C, typename T, bool UPDATE>
struct ColSource {
  static constexpr bool kWriteBack = UPDATE;
  const C* __restrict__ in;
  const C* __restrict__ pold;
  C* __restrict__ pnew;
  const int* off;
  T beta;
  int inner;        // row stride
  int half, M, width;
  __device__ __forceinline__ int index(int t, int n, bool& ok) const {
    const int r = n <= half ? n : (n >= M - half ? n - M : M);   // row offset from the centre
    ok = r != M && t < width;
    return off[t] + (r + half) * inner;
  }
  __device__ __forceinline__ C operator()(int t, int n) const {
    bool ok;
    const int idx = index(t, n, ok);
    C v = mk(T(0), T(0));
    if (ok) {
      v = in[idx];
      if constexpr (UPDATE) {
        const C po = pold[idx];
        v = mk(v.x + beta * po.x, v.y + beta * po.y);
      }
    }
    return v;
  }
  __device__ __forceinline__ void write_back(int t, int n, C v) const {
    bool ok;
    const int idx = index(t, n, ok);
    if (ok) pnew[idx] = v;
  }
};

template <int TW, int SIGN, int MODE, int M>
__device__ __forceinline__ void col_body(const ColArgs& a, const CtTables& pl, int64_t bid) {
  using T = float;
  using C = float2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* buf = reinterpret_cast<C*>(smem_raw);

  // TW consecutive columns of the flattened (outer, inner) range, so that no CTA
  // is spent on the ragged end of each outer index
  __shared__ int s_in[TW], s_out[TW];
  const int64_t ncols = a.outer * a.inner;
  const int64_t g0 = bid * TW;
  const int width = static_cast<int>(ncols - g0 < TW ? ncols - g0 : TW);
  const int64_t rows_in = SIGN > 0 ? a.Lin : M;
  const int64_t rows_out = SIGN > 0 ? M : a.Lout;
  if (threadIdx.x < TW) {
    const int64_t g = g0 + (static_cast<int>(threadIdx.x) < width ? threadIdx.x : width - 1);
    const int64_t oo = g / a.inner, jj = g - oo * a.inner;
    s_in[threadIdx.x] = static_cast<int>(oo * rows_in * a.inner + jj);
    s_out[threadIdx.x] = static_cast<int>(oo * rows_out * a.inner + jj);
  }
  grid_wait();
  if (a.st != nullptr && a.st->done != RUNNING) return;
  __syncthreads();
  const C* __restrict__ tw = pl.tw;
  const C* __restrict__ in = after_wait(static_cast<const C*>(a.in));
  C* __restrict__ out = static_cast<C*>(a.out);

  if constexpr (SIGN > 0) {
    // The transform reads its input rows straight from global memory in its first
    // pass (input n of line t is row i(n) of the tile, zero outside the padded
    // range; p = r + beta p_old is formed and written back on the way).
    const int Lin = a.Lin;
    const int half = (Lin - 1) / 2;
    T beta = T(0);
    const C* pold = nullptr;
    C* pnew = nullptr;
    if constexpr (MODE == COL_PUPDATE) {
      beta = static_cast<T>(a.st->beta);
      pold = after_wait(static_cast<const C*>(a.pold));
      pnew = static_cast<C*>(a.pnew);
    }
    ColSource<C, T, MODE == COL_PUPDATE> src{in, pold, pnew, s_in, beta, static_cast<int>(a.inner), half, M, width};
    fft_dit_ct_src<+1, TW, col_threads<TW, M, MODE>(), M>(buf, tw, src);
    for (int u = threadIdx.x; u < M * TW; u += blockDim.x) {
      const int t = u % TW;
      const int m = u / TW;
      if (t < width) out[s_out[t] + m * static_cast<int>(a.inner)] = buf[m * TW + t];
    }
  } else {
    // natural-order input copied in, the last pass hands the kept frequencies
    // (scaled by 1/M) straight to global memory
    for (int u = threadIdx.x; u < M * TW; u += blockDim.x) {
      const int t = u % TW;
      const int m = u / TW;
      if (t < width) cp_async<sizeof(C)>(buf + u, in + (s_in[t] + m * static_cast<int>(a.inner)));
      else buf[u] = mk(T(0), T(0));
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    const int Lout = a.Lout;
    const int half = (Lout - 1) / 2;
    const T inv = T(1) / T(M);
    auto snk = [&](int t, int n, C v) {
      const int i = n <= half ? n + half : (n >= M - half ? n - M + half : -1);
      if (i >= 0 && t < width) out[s_out[t] + i * static_cast<int>(a.inner)] = inv * v;
    };
    fft_dif_ct_snk<-1, TW, col_threads<TW, M, MODE>(), M>(buf, tw, snk);
  }
}

template <int TW, int SIGN, int MODE, int M>
__global__ void __launch_bounds__(col_threads<TW, M, MODE>(), col_min_blocks<TW, M, MODE>())
    col_kernel(ColArgs a, CtTables pl) {
  col_body<TW, SIGN, MODE, M>(a, pl, blockIdx.x);
}

template <int TW, int SIGN, int MODE, int M>
inline ghb_status launch_col_t(const ColArgs& a, const CtTables& pl, cudaStream_t s) {
  const size_t smem = col_smem_bytes(M, TW, sizeof(float2));
  static std::atomic<unsigned long long> attr_mask{0};
  TRY_STATUS(ensure_dyn_smem(col_kernel<TW, SIGN, MODE, M>, 220 * 1024, attr_mask));
  const int64_t grid = (a.outer * a.inner + TW - 1) / TW;
  if (a.outer * std::max<int64_t>(std::max<int64_t>(a.Lin, a.Lout), M) * a.inner >= (int64_t(1) << 31)) {
    set_error("column pass operand of 2^31 entries or more");
    return GHB_ERR_INVALID;
  }
  return launch_chained(col_kernel<TW, SIGN, MODE, M>, grid, col_threads<TW, M, MODE>(), smem, s, a, pl);
}

// ---------------------------------------------------------------------------
// row pass
// ---------------------------------------------------------------------------
struct LineDesc {
  int64_t row;
  int field;
  int comp;
  int valid;
};

// Field f of a row pass.  Selects rather than an index into the argument's
// array: a run-time index into a kernel parameter makes the compiler copy the
// whole argument to local memory and load the pointer from there (the FP32
// last-axis pass at M = 4374: 164 -> 145 us without that copy and without
// the per-entry line masks of its staged spectra).
__device__ __forceinline__ void* row_field(const RowArgs& a, int f) {
  return f == 0 ? a.t[0] : (f == 1 ? a.t[1] : a.t[2]);
}

// Threads of a last-axis CTA.  A_M is read from global memory in the fused pass
// (coalesced: a warp's threads hold consecutive entries) instead of staged,
// which leaves shared memory for a fourth CTA per SM; a radix-27 pass at M = 4374
// has 162 butterflies per line.  At M = 4374: 173 us per launch against 184 us
// with the staged A_M and 256 threads; at M = 270 (15 lines per CTA): 300 us
// against 334 us.
constexpr int kRowThreads = 192;

// Operator pass with staged inputs.  The CTA loops over row groups; the next
// group's half spectra are copied asynchronously into a staging area while the
// current group is transformed:
//
//   smem = [ transform buffer | staged half spectra [2 NL][H] ]
//
// Staged half spectra: the two real lines of complex line j side by side,
// entry (j, k) at pair index j * row_pair_stride(H) + k (an odd stride, so that
// threads of consecutive lines reading the same k fall on different banks).
__host__ __device__ inline int row_pair_stride(int H) { return H | 1; }
__host__ __device__ inline size_t row_buf_elems(int M, int NL) {   // rounded to 16 bytes
  return (padded_elems<float2>(static_cast<size_t>(M) * NL) + 1) & ~static_cast<size_t>(1);
}
template <int NL>
__host__ __device__ inline size_t row_staged_smem(int M, int H) {
  return (row_buf_elems(M, NL) + static_cast<size_t>(2 * NL) * row_pair_stride(H)) * sizeof(float2);
}

// Input of the size-specialised last-axis transforms: entry n of complex line
// j is the Hermitian completion of the two staged half spectra X0, X1 of its
// real lines (X(k), k = 0 .. H-1; line pairs at stride SH):
//     Z(n) = X0(n) + i X1(n)                      n < H,
//     Z(n) = conj X0(M-n) + i conj X1(M-n)        n > M - H,
//     0                                           otherwise.
// With RANGED, ranged() decides for a whole range of n at once (see
// ct_ranged): in the first pass at M = 4374, N = 2187 every range but two lies
// entirely below H, entirely above M - H or entirely in the zeros.  Measured:
// 209 -> 204 us at M = 270, but 144 -> 148 us at M = 4374, which therefore keeps
// the test per entry.
template <typename C, typename Pair, bool RANGED>
struct RowSource {
  static constexpr bool kRanged = RANGED;
  const Pair* spair;
  int SH, H, M;
  __device__ __forceinline__ C lo(int j, int k) const {
    const Pair v = spair[j * SH + k];   // both real lines in one load
    return mk(v.a.x - v.b.y, v.a.y + v.b.x);
  }
  __device__ __forceinline__ C hi(int j, int k) const {
    const Pair v = spair[j * SH + k];
    return mk(v.a.x + v.b.y, v.b.x - v.a.y);
  }
  __device__ __forceinline__ C operator()(int j, int n) const {
    using T = decltype(C{}.x);
    const bool l = n < H, h = n > M - H;
    const int k = l ? n : M - n;
    C A = mk(T(0), T(0)), B = mk(T(0), T(0));
    if (l || h) {
      const Pair v = spair[j * SH + k];
      A = v.a;
      B = v.b;
    }
    return l ? mk(A.x - B.y, A.y + B.x) : mk(A.x + B.y, B.x - A.y);
  }
  __device__ __forceinline__ C ranged(int j, int nb, int n0, int span) const {
    using T = decltype(C{}.x);
    if (n0 + span - 1 < H) return lo(j, nb + n0);
    if (n0 > M - H) return hi(j, M - n0 - nb);
    if (n0 >= H && n0 + span - 1 <= M - H) return mk(T(0), T(0));
    return (*this)(j, nb + n0);
  }
};

template <int NL, int M>
__device__ __forceinline__ void row_matvec_staged(const RowArgs& a, const CtTables& pl, int rows_per_cta,
                                                  int64_t bid, int64_t nb) {
  using T = float;
  using C = float2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ LineDesc ld[2 * NL], ldn[2 * NL];   // this group's lines, the next group's
  __shared__ int2 lrow[NL];                      // offsets in A_M of each complex line's two rows
  grid_wait();
  if (a.st != nullptr && a.st->done != RUNNING) return;

  const int H = a.H;
  const int per_row = a.nfields * a.ncomp;
  const int nrl = rows_per_cta * per_row;
  const int64_t groups = (a.rows + rows_per_cta - 1) / rows_per_cta;
  C* buf = reinterpret_cast<C*>(smem_raw);
  C* sin = buf + row_buf_elems(M, NL);
  const int SH = row_pair_stride(H);
  struct alignas(2 * sizeof(C)) Pair {
    C a, b;
  };
  const Pair* spair = reinterpret_cast<const Pair*>(sin);
  const C* __restrict__ tw = pl.tw;
  const int* __restrict__ perm = pl.perm;
  const T* __restrict__ am = static_cast<const T*>(a.a);

  auto desc = [&](int64_t grp, int rho) {
    LineDesc d;
    d.row = grp * rows_per_cta + rho / per_row;
    d.field = (rho / a.ncomp) % a.nfields;
    d.comp = rho % a.ncomp;
    d.valid = (rho < nrl) && (d.row < a.rows);
    return d;
  };
  // Copies of the half spectra of the lines described by L[0 .. 2NL) into the
  // staging area; a line that is not valid (past the last row) gets zeros,
  // so that the transforms read the staged pairs without masks.  Long rows
  // (H >= the block): line by line, the block striding over k.  Short rows:
  // one flat loop over (line, k), the line and k of a thread advanced by the
  // block size each step (no division per entry).
  auto issue_from = [&](const LineDesc* L) {
    if (H >= static_cast<int>(blockDim.x)) {
#pragma unroll 1
      for (int rho = 0; rho < 2 * NL; ++rho) {
        const LineDesc d = L[rho];
        C* dst = sin + (rho >> 1) * 2 * SH + (rho & 1);
        if (!d.valid) {
          for (int k = threadIdx.x; k < H; k += blockDim.x) dst[2 * k] = mk(T(0), T(0));
          continue;
        }
        const C* src = static_cast<const C*>(row_field(a, d.field)) + d.comp * a.comp_stride + d.row * H;
        for (int k = threadIdx.x; k < H; k += blockDim.x) cp_async<sizeof(C)>(dst + 2 * k, src + k);
      }
      return;
    }
    const int step_r = static_cast<int>(blockDim.x) / H, step_k = static_cast<int>(blockDim.x) - step_r * H;
    int rho = static_cast<int>(threadIdx.x) / H;
    int k = static_cast<int>(threadIdx.x) - rho * H;
    while (rho < 2 * NL) {
      const LineDesc d = L[rho];
      C* dst = sin + ((rho >> 1) * SH + k) * 2 + (rho & 1);
      if (d.valid)
        cp_async<sizeof(C)>(dst, static_cast<const C*>(row_field(a, d.field)) + d.comp * a.comp_stride + d.row * H + k);
      else
        *dst = mk(T(0), T(0));
      rho += step_r;
      k += step_k;
      if (k >= H) {
        k -= H;
        ++rho;
      }
    }
  };
  int64_t grp = bid;
  if (grp < groups) {
    if (threadIdx.x < 2 * NL) ldn[threadIdx.x] = desc(grp, threadIdx.x);
    __syncthreads();
    issue_from(ldn);
    cp_async_commit();
    __syncthreads();   // ldn is rewritten at the top of the loop
  }
  for (; grp < groups; grp += nb) {
    // every thread has issued the copies of ldn's lines (barriers since then)
    if (threadIdx.x < 2 * NL) {
      ld[threadIdx.x] = desc(grp, threadIdx.x);
      ldn[threadIdx.x] = desc(grp + nb, threadIdx.x);
    }
    if (threadIdx.x < NL) {
      const LineDesc d0 = desc(grp, 2 * threadIdx.x), d1 = desc(grp, 2 * threadIdx.x + 1);
      lrow[threadIdx.x] =
          make_int2(d0.valid ? static_cast<int>(d0.row * M) : 0, d1.valid ? static_cast<int>(d1.row * M) : 0);
    }
    cp_async_wait<0>();          // spectra(g) are in
    __syncthreads();

    // the staged pairs hold zeros for a line that is not valid
    constexpr bool ranged = M == 72 || M == 135 || M == 270;
    const RowSource<C, Pair, ranged> src{spair, SH, H, M};
    // multiply by A_M between the transforms, in registers; a line that is not
    // valid reads row 0 (in bounds, finite) and is not stored; its zero input
    // keeps the other line of the pair exact
    auto mul = [&](int j, int m, C z) -> C {
      const int2 ro = lrow[j];
      return mk(__ldg(&am[ro.x + m]) * z.x, __ldg(&am[ro.y + m]) * z.y);
    };
    auto after_first = [&]() {   // the staged spectra are read: stage the next group's
      if (grp + nb < groups) issue_from(ldn);
      cp_async_commit();
    };
    auto nothing = [&]() {};
    ct_inverse_scale_forward<+1, -1, NL, kRowThreads, M>(buf, tw, src, mul, after_first, nothing,
                                                         nothing);   // ends with a barrier
    const T sc = T(0.5) / T(M);
    for (int u = threadIdx.x; u < NL * H; u += blockDim.x) {
      const int j = (NL == 1) ? 0 : u % NL;
      const int k = (NL == 1) ? u : u / NL;
      const LineDesc d0 = ld[2 * j], d1 = ld[2 * j + 1];
      const C W = buf[__ldg(&perm[k]) * NL + j];
      const C Wm = buf[__ldg(&perm[k == 0 ? 0 : M - k]) * NL + j];
      if (d0.valid)
        static_cast<C*>(row_field(a, d0.field))[d0.comp * a.comp_stride + d0.row * H + k] =
            mk(sc * (W.x + Wm.x), sc * (W.y - Wm.y));
      if (d1.valid)
        static_cast<C*>(row_field(a, d1.field))[d1.comp * a.comp_stride + d1.row * H + k] =
            mk(sc * (W.y + Wm.y), sc * (Wm.x - W.x));
    }
    __syncthreads();
  }
  cp_async_wait<0>();
}

// at most 85 registers so that four CTAs share an SM
template <int NL, int M>
__global__ void __launch_bounds__(kRowThreads, 4) row_kernel_staged(RowArgs a, CtTables pl, int rows_per_cta) {
  row_matvec_staged<NL, M>(a, pl, rows_per_cta, blockIdx.x, gridDim.x);
}

template <int NL, int M>
inline ghb_status launch_row_t(const RowArgs& a, const CtTables& pl, int rows_per_cta, cudaStream_t s) {
  const int64_t groups = (a.rows + rows_per_cta - 1) / rows_per_cta;
  const size_t smem = row_staged_smem<NL>(M, a.H);
  if (smem > 200 * 1024) {
    set_error("row transform too large for one CTA: M=" + std::to_string(M));
    return GHB_ERR_INVALID;
  }
  // persistent grid: as many CTAs as fit on the device at once (the occupancy
  // per device and staging size, kept per device)
  static std::atomic<unsigned long long> staged_mask{0};
  TRY_STATUS(ensure_dyn_smem(row_kernel_staged<NL, M>, 200 * 1024, staged_mask));
  struct Occ {
    size_t smem;
    int per_sm, sms;
  };
  static std::mutex occ_mutex;
  static Occ occ[64] = {};
  int dev = 0;
  GHB_CUDA_TRY(cudaGetDevice(&dev));
  Occ o{0, 0, 0};
  {
    std::lock_guard<std::mutex> lock(occ_mutex);
    if (dev < 64) o = occ[dev];
  }
  if (o.smem != smem) {
    o.smem = smem;
    GHB_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o.per_sm, row_kernel_staged<NL, M>, kRowThreads, smem));
    GHB_CUDA_TRY(cudaDeviceGetAttribute(&o.sms, cudaDevAttrMultiProcessorCount, dev));
    std::lock_guard<std::mutex> lock(occ_mutex);
    if (dev < 64) occ[dev] = o;
  }
  int64_t grid = static_cast<int64_t>(o.per_sm > 0 ? o.per_sm : 1) * o.sms;
  if (grid > groups) grid = groups;
  if (grid < 1) grid = 1;
  return launch_chained(row_kernel_staged<NL, M>, grid, kRowThreads, smem, s, a, pl, rows_per_cta);
}

// Size-specialised operator passes of transform length M (instantiated in the
// ct_*.cu units).
template <int M>
ghb_status launch_col_ct_m(int sign, int mode, const ColArgs& a, const CtTables& pl, cudaStream_t s) {
  constexpr int TW = col_tile_width(M, sizeof(float2));
  if (sign < 0) return launch_col_t<TW, -1, COL_PLAIN, M>(a, pl, s);
  return mode == COL_PUPDATE ? launch_col_t<TW, +1, COL_PUPDATE, M>(a, pl, s)
                             : launch_col_t<TW, +1, COL_PLAIN, M>(a, pl, s);
}
// Interleaved complex lines that give every thread a butterfly in every pass,
// for PER_ROW real lines per row (2 in 2-D, 3 in 3-D: a multiple of 3 so that
// the lines make whole rows), at most 32.
// In 3-D the counts below were chosen by a sweep of 6 .. 24 lines on GB300
// (one d = 3 operator application per setting): lines that make each pass
// about one full round of the block, with four CTAs per SM, beat the rule
// (M = 270: 12 lines, 221 against 242 us; M = 162: 18 lines, 55.8 against 61.7 us;
// M = 135: 12 lines; M = 72: 18 lines).
template <int M, int PER_ROW>
__host__ __device__ constexpr int ct_fill_lines() {
  if (PER_ROW == 3) {
    if (M == 270 || M == 135) return 12;
    if (M == 162 || M == 72) return 18;
  }
  int nl = (kRowThreads + ct_min_units<M>() - 1) / ct_min_units<M>();
  if (nl > 32) nl = 32;
  if (PER_ROW == 3) nl = 3 * ((nl + 2) / 3);
  if (nl > 32) nl = 30;
  return nl;
}

template <int M>
ghb_status launch_row_ct_m(int NL, const RowArgs& a, const CtTables& pl, int rows_per_cta, cudaStream_t s) {
  // Short transforms (the 3-D double grids, 2-D ones up to M = 486) leave
  // most threads without a butterfly at one to three lines per CTA: take as
  // many rows as fill the CTA when the row rule leaves more than half of the
  // threads idle and the staging still fits (at M = 1458, where two lines
  // leave 44 % idle, four lines measured slower: 32.7 against 28.4 us).
  const int per_row = a.nfields * a.ncomp;
  if ((per_row == 2 || per_row == 3) && ct_min_units<M>() * NL * 2 < kRowThreads) {
    constexpr int NL2 = ct_fill_lines<M, 2>(), NL3 = ct_fill_lines<M, 3>();
    const int want = per_row == 2 ? NL2 : NL3;
    const int rows = 2 * want / per_row;
    const size_t smem = per_row == 2 ? row_staged_smem<NL2>(M, a.H) : row_staged_smem<NL3>(M, a.H);
    if (want > NL && smem <= 200 * 1024) {
      if (per_row == 2) return launch_row_t<NL2, M>(a, pl, rows, s);
      return launch_row_t<NL3, M>(a, pl, rows, s);
    }
  }
  switch (NL) {
    case 1: return launch_row_t<1, M>(a, pl, rows_per_cta, s);
    case 2: return launch_row_t<2, M>(a, pl, rows_per_cta, s);
    case 3: return launch_row_t<3, M>(a, pl, rows_per_cta, s);
    default: break;
  }
  set_error("internal: unsupported row-pass line count");
  return GHB_ERR_INVALID;
}

}  // namespace ghb
