// FP32 transform passes for run-time plans (fft_rt.cuh): the column pass and the
// operator's last-axis pass, every length.  Lines are held whole in shared
// memory; positions and passes are laid out as in the FP64 passes (FxPass).
#pragma once

#include "fft_rt.cuh"
#include "ghb_internal.cuh"
#include "launch_util.cuh"

namespace ghb {

// Largest block: 24 warps of up to 80 registers (a group of 16 takes 32), as one
// CTA or as several smaller ones.
constexpr int kRtThreads = 768;
// The last-axis and the batched column kernels are also compiled for 64 registers,
// 32 warps an SM: they spill a little, and gain where more warps than 24 an SM have
// work at once.  N = 1023 operator 68 -> 66.5 us, N = 1215 115 -> 112.7, 64 mixed
// microstructures 236 -> 227 ms; with fewer, 80 registers are better (N = 405 32.2
// against 32.7 us, N = 511 bound pair 20.4 against 20.8 ms), and for single column
// passes always (N = 1023 operator 66.5 against 71.9).
constexpr int kRtManyThreads = 1024;
bool rt_many_warps(int64_t blocks, int threads);   // passes.cu
constexpr int kRtMaxLines = 32;

struct RtShared {
  FxPass p[kFxPasses];
  int np;
};
__device__ __forceinline__ void rt_load_plan(RtShared& sh, const FxPlan& f) {
  const int n = f.np * static_cast<int>(sizeof(FxPass) / sizeof(int));
  const int* src = reinterpret_cast<const int*>(f.p);
  int* dst = reinterpret_cast<int*>(sh.p);
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
  if (threadIdx.x == 0) sh.np = f.np;
}

// Unit t of a pass over `lines` lines (line q at buf + q ls).  QFAST: lines
// alternate fastest (columns: a row's columns are neighbours in memory; lines is
// a power of two), else units do (rows).
template <bool FIRST, bool QFAST>
__device__ __forceinline__ RtUnit rt_unit(float2* buf, int ls, int lines, const FxPass& P, const FxPlan& f, int t) {
  RtUnit u;
  int unit;
  if (QFAST) {
    u.q = t & (lines - 1);
    unit = t >> (31 - __clz(lines));
  } else {
    u.q = static_cast<int>(fdiv(static_cast<unsigned>(t), P.ulines));
    unit = t - u.q * P.units;
  }
  int pos;
  if (FIRST) {
    u.p = 0;
    u.r = unit;
    pos = __ldg(&f.perm[unit]);
  } else {
    const int b = static_cast<int>(fdiv(static_cast<unsigned>(unit), P.ulp));
    u.p = unit - b * P.lp;
    u.r = 0;
    pos = __ldg(&f.nat[b * (P.lp * P.R) + u.p]);
  }
  u.base = buf + u.q * ls + pos;
  return u;
}

template <int SIGN, bool DIT, bool FIRST, bool QFAST, typename Src, typename Snk>
__device__ __forceinline__ void rt_pass(float2* buf, int ls, int lines, const FxPass& P, const FxPlan& f, int M,
                                        const float2* __restrict__ tw, const Src& src, const Snk& snk) {
  const int total = P.units * lines;
  for (int t = threadIdx.x; t < total; t += blockDim.x) {
    const RtUnit u = rt_unit<FIRST, QFAST>(buf, ls, lines, P, f, t);
    rt_run_unit<SIGN, DIT, FIRST>(P, u, M, tw, src, snk);
  }
}

// A whole transform of np >= 1 passes from src to snk.  No barrier before or after.
template <int SIGN, bool QFAST, typename Src, typename Snk>
__device__ __forceinline__ void rt_transform(float2* buf, int ls, int lines, const RtShared& sh, const FxPlan& f, int M,
                                             const float2* __restrict__ tw, const Src& src, const Snk& snk) {
  constexpr bool DIT = SIGN > 0;
  const int np = sh.np;
  if (np == 1) {
    rt_pass<SIGN, DIT, true, QFAST>(buf, ls, lines, sh.p[0], f, M, tw, src, snk);
    return;
  }
  if (DIT) rt_pass<SIGN, DIT, true, QFAST>(buf, ls, lines, sh.p[0], f, M, tw, src, RtMem());
  else rt_pass<SIGN, DIT, false, QFAST>(buf, ls, lines, sh.p[np - 1], f, M, tw, src, RtMem());
  for (int k = 1; k < np - 1; ++k) {
    __syncthreads();
    rt_pass<SIGN, DIT, false, QFAST>(buf, ls, lines, sh.p[DIT ? k : np - 1 - k], f, M, tw, RtMem(), RtMem());
  }
  __syncthreads();
  if (DIT) rt_pass<SIGN, DIT, false, QFAST>(buf, ls, lines, sh.p[np - 1], f, M, tw, RtMem(), snk);
  else rt_pass<SIGN, DIT, true, QFAST>(buf, ls, lines, sh.p[0], f, M, tw, RtMem(), snk);
}

// ---------------------------------------------------------------------------
// column pass: TW (a power of two) neighbouring columns of the flattened (outer,
// inner) range; a thread always handles the same column.  Input rows are read
// by the first pass (inverse: zero-padded, p = r + beta p_old formed and written
// back), the last pass stores the output rows.
// ---------------------------------------------------------------------------
template <bool UPDATE>
struct RtColIn {
  static constexpr bool kUpdate = UPDATE;
  const float2 *in, *old;
  float2* upd;
  float beta;
  int inner;            // row stride (the rows of one outer index hold fewer than 2^31 entries)
  int half, wrap;       // rows: n <= half -> n + half, n >= wrap -> n - wrap (wrap = M - half)
  bool on;
  __device__ __forceinline__ int row(int n) const { return n <= half ? n + half : (n >= wrap ? n - wrap : -1); }
  __device__ __forceinline__ float2 operator()(int, int n) const {
    const int i = row(n);
    float2 a = make_float2(0.0f, 0.0f);
    if (i >= 0 && on) {
      a = in[i * inner];
      if (UPDATE) {
        const float2 o = old[i * inner];
        a = make_float2(a.x + beta * o.x, a.y + beta * o.y);
      }
    }
    return a;
  }
  __device__ __forceinline__ void store(int, int n, float2 v) const {
    const int i = row(n);
    if (i >= 0 && on) upd[i * inner] = v;
  }
};

template <int SIGN, bool UPDATE>
__device__ __forceinline__ void rt_col_body(const ColArgs& a, const FxPlan& f, int TW, int64_t bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* buf = reinterpret_cast<float2*>(smem_raw);
  __shared__ RtShared sh;
  const int M = f.M;
  rt_load_plan(sh, f);
  const int t = threadIdx.x & (TW - 1);
  const int64_t ncols = a.outer * a.inner;
  const int inner = static_cast<int>(a.inner);
  const int64_t g = bid * TW + t;
  const bool on = g < ncols;
  const int64_t o = on ? g / a.inner : 0, j = on ? g - o * a.inner : 0;
  const int Lin = SIGN > 0 ? a.Lin : M, Lout = SIGN > 0 ? M : a.Lout;
  const int64_t off = o * Lin * a.inner + j;
  grid_wait();
  if (a.st != nullptr && a.st->done != RUNNING) return;
  RtColIn<UPDATE> src{};
  src.in = static_cast<const float2*>(a.in) + off;
  src.inner = inner;
  src.on = on;
  src.half = (Lin - 1) / 2;
  src.wrap = M - src.half;
  if (UPDATE) {
    src.beta = static_cast<float>(a.st->beta);
    src.old = static_cast<const float2*>(a.pold) + off;
    src.upd = static_cast<float2*>(a.pnew) + off;
  }
  float2* out = static_cast<float2*>(a.out) + o * Lout * a.inner + j;
  const int hout = (Lout - 1) / 2;
  const float inv = 1.0f / static_cast<float>(M);
  const auto snk = [&](int, int n, float2 v) {
    int i = n;
    if (SIGN < 0) {
      i = n <= hout ? n + hout : (n >= M - hout ? n - M + hout : -1);
      v = inv * v;
    }
    if (i >= 0 && on) out[i * inner] = v;
  };
  const auto fwd = [&](int, int n) {   // forward input: every row
    return on ? src.in[n * inner] : make_float2(0.0f, 0.0f);
  };
  __syncthreads();   // plan in place
  if (sh.np == 0) {   // M = 1
    if (threadIdx.x < TW) {
      const float2 v = src(t, 0);
      if (UPDATE) src.store(t, 0, v);
      snk(t, 0, v);
    }
    return;
  }
  const int ls = column_stride(f.ls, TW, sizeof(float2));
  if constexpr (SIGN > 0) rt_transform<+1, true>(buf, ls, TW, sh, f, M, f.tw32, src, snk);
  else rt_transform<-1, true>(buf, ls, TW, sh, f, M, f.tw32, fwd, snk);
}

// ---------------------------------------------------------------------------
// last-axis pass of the operator: complex lines z = u + i v of two real lines
// (field component c of row r is real line r ncomp + c).
// ---------------------------------------------------------------------------
struct RtLine {
  int64_t off[2];     // first entry of the real lines
  int64_t row[2];     // element offset of their rows of A_M
  int valid;
};

__device__ __forceinline__ void rt_row_body(const RowArgs& a, const FxPlan& f, int rows_per_cta, int lines,
                                            int64_t bid, int64_t nb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* buf = reinterpret_cast<float2*>(smem_raw);
  __shared__ RtShared sh;
  __shared__ RtLine ld[kRtMaxLines];
  const int M = f.M, H = a.H, ls = f.ls;
  const int nrl = rows_per_cta * a.ncomp;
  const int64_t groups = (a.rows + rows_per_cta - 1) / rows_per_cta;
  const int* __restrict__ perm = f.perm;
  const float2* __restrict__ tw = f.tw32;
  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);
  const int nwarp = blockDim.x >> 5;
  const int segs = nwarp > lines ? nwarp / lines : 1;
  float2* data = static_cast<float2*>(a.t[0]);
  const float* __restrict__ am = static_cast<const float*>(a.a);
  rt_load_plan(sh, f);
  grid_wait();
  if (a.st != nullptr && a.st->done != RUNNING) return;

  // input n of line q: Z(n) = X0(n) + i X1(n) below H, conj X0 + i conj X1 at M - n
  // above M - H, zero between
  const auto src = [&](int q, int n) {
    const RtLine& d = ld[q];
    const bool l = n < H, h = n > M - H;
    const int k = l ? n : M - n;
    float2 A = make_float2(0.0f, 0.0f), B = A;
    if (l || h) {
      if (d.valid & 1) A = data[d.off[0] + k];
      if (d.valid & 2) B = data[d.off[1] + k];
    }
    return l ? make_float2(A.x - B.y, A.y + B.x) : make_float2(A.x + B.y, B.x - A.y);
  };
  const auto mul = [&](int q, int m, float2 v) {
    const RtLine& d = ld[q];
    return make_float2(__ldg(&am[d.row[0] + m]) * v.x, __ldg(&am[d.row[1] + m]) * v.y);
  };

  for (int64_t grp = bid; grp < groups; grp += nb) {
    if (threadIdx.x < lines) {
      RtLine d;
      d.valid = 0;
      for (int r = 0; r < 2; ++r) {
        const int rho = 2 * threadIdx.x + r;
        const int64_t row = grp * rows_per_cta + rho / a.ncomp;
        const bool here = rho < nrl && row < a.rows;
        if (here) d.valid |= 1 << r;
        d.row[r] = here ? row * M : 0;   // a line that is not there reads row 0 and is not stored
        d.off[r] = (rho % a.ncomp) * a.comp_stride + row * H;
      }
      ld[threadIdx.x] = d;
    }
    __syncthreads();
    const int np = sh.np;
    if (np == 0) {   // M = 1
      if (threadIdx.x < lines) buf[threadIdx.x * ls] = mul(threadIdx.x, 0, src(threadIdx.x, 0));
    } else {
      rt_pass<+1, true, true, false>(buf, ls, lines, sh.p[0], f, M, tw, src, RtMem());
      __syncthreads();
      for (int k = 1; k < np - 1; ++k) {
        rt_pass<+1, true, false, false>(buf, ls, lines, sh.p[k], f, M, tw, RtMem(), RtMem());
        __syncthreads();
      }
      if (np > 1) {
        const FxPass P = sh.p[np - 1];
        for (int t = threadIdx.x; t < P.units * lines; t += blockDim.x)
          rt_run_fused(P, rt_unit<false, false>(buf, ls, lines, P, f, t), M, tw, mul);
      } else {   // one pass: the line is a group, in natural order after the inverse
        for (int t = threadIdx.x; t < M * lines; t += blockDim.x) {
          const int q = t / M, m = t - q * M;
          float2& v = buf[q * ls + m];
          v = mul(q, m, v);
        }
        __syncthreads();
        rt_pass<-1, false, true, false>(buf, ls, lines, sh.p[0], f, M, tw, RtMem(), RtMem());
      }
      for (int k = np - 2; k >= 0; --k) {
        __syncthreads();
        if (k > 0) rt_pass<-1, false, false, false>(buf, ls, lines, sh.p[k], f, M, tw, RtMem(), RtMem());
        else rt_pass<-1, false, true, false>(buf, ls, lines, sh.p[0], f, M, tw, RtMem(), RtMem());
      }
    }
    __syncthreads();

    const float sc = 0.5f / static_cast<float>(M);
    for (int idx = warp; idx < lines * segs; idx += nwarp) {
      const int q = idx / segs, k0 = (idx - q * segs) * 32 + lane;
      const RtLine& d = ld[q];
      const float2* line = buf + q * ls;
#pragma unroll 4
      for (int k = k0; k < H; k += 32 * segs) {
        const float2 W = line[__ldg(&perm[k])];
        const float2 V = line[__ldg(&perm[k == 0 ? 0 : M - k])];
        // X0 = (W + conj V)/2, X1 = (W - conj V)/(2 i)
        if (d.valid & 1) data[d.off[0] + k] = make_float2(sc * (W.x + V.x), sc * (W.y - V.y));
        if (d.valid & 2) data[d.off[1] + k] = make_float2(sc * (W.y + V.y), sc * (V.x - W.x));
      }
    }
    __syncthreads();
  }
}

// Launch shapes (passes.cu) and launchers (rt_col.cu, rt_row.cu).
int rt_col_tile(int M, int ls, int64_t columns);
int rt_threads(int M, int lines, int ls);
// want: 0 = lines by size, 1 / 2 = the least rows once or twice
void rt_row_shape(int ncomp, int M, int ls, int64_t rows, int want, int* rows_per_cta, int* lines);
ghb_status launch_rt_col(int sign, const ColArgs& a, const FxPlan& f, int TW, cudaStream_t s);
ghb_status launch_rt_col_batch(int sign, bool update, const ColItem* items, int n, int64_t blocks, size_t smem,
                               int threads, cudaStream_t s);
ghb_status launch_rt_row(const RowArgs& a, const FxPlan& f, int rows_per_cta, int lines, cudaStream_t s);
ghb_status launch_rt_row_batch(const RowItem* items, int n, int64_t blocks, size_t smem, int threads,
                               cudaStream_t s);

}  // namespace ghb
