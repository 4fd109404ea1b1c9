// FP64 transform passes of the double-grid operator on the fixed-point
// transform (fft_fx.cuh): the column pass and the last-axis pass with the same
// inputs, outputs and modes as the FP32 templates of passes_impl.cuh, for every
// supported length (one run-time plan; no size-specialised kernels).
//
// Bound by integer issue (53 % of the ALU pipe's cycles, 2.1 instructions a
// clock): about 65 instructions per entry and pass of nine entries a thread
// (radix 3 x 3), a third of the pass's time in conversions and the multiply.
// One CTA holds its lines whole in shared memory, one after the other.
// Measured against the FP64-pipe kernels these replace (N = 2187, M = 4374):
// last axis 4267 -> 961 us, axis 1 1048 / 1047 -> 331 / 304 us, one operator
// application 6.50 -> 1.73 ms; d = 3, N = 63 x 99 x 77 2.51 -> 0.54 ms; N = 315 x
// 517 354 -> 98 us.
#pragma once

#include <algorithm>

#include "fft_fx.cuh"
#include "ghb_internal.cuh"
#include "launch_util.cuh"
#include "reduce.cuh"

namespace ghb {

constexpr int kFxMaxLines = 32;
// Largest block: 24 warps of up to 80 registers (nine entries a thread take 36
// of them), as one CTA or as three of 256 threads.
constexpr int kFxThreads = 768;
constexpr int kFxBlocks = 1;

// Shared state of a CTA: the plan, and per line the exponents and the
// magnitudes after each pass (slot k: before the k-th pass of the sequence).
struct FxShared {
  FxPass p[kFxPasses];
  int np;
  int mag[2 * kFxPasses + 2][kFxMaxLines];
  int emax[kFxMaxLines];    // largest |word| of the line's doubles, then its biased exponent
  int wmax[kFxMaxLines];    // the same of the line after the multiply
};

__device__ __forceinline__ void fx_load_plan(FxShared& sh, const FxPlan& f) {
  const int n = f.np * static_cast<int>(sizeof(FxPass) / sizeof(int));
  const int* src = reinterpret_cast<const int*>(f.p);
  int* dst = reinterpret_cast<int*>(sh.p);
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
  if (threadIdx.x == 0) sh.np = f.np;
}

__device__ __forceinline__ void fx_clear_lines(FxShared& sh) {
  for (int i = threadIdx.x; i < (2 * kFxPasses + 2) * kFxMaxLines; i += blockDim.x) (&sh.mag[0][0])[i] = 0;
  if (threadIdx.x < kFxMaxLines) sh.emax[threadIdx.x] = sh.wmax[threadIdx.x] = 0;
}

// Shift before the pass in slot k (bits: what it admits); the first pass after
// a conversion needs none.
__device__ __forceinline__ int fx_shift_of(const FxShared& sh, int k, int k0, int bits, int line) {
  if (k == k0) return 0;
  return bits - fx_bitlen(sh.mag[k][line]);
}

// The passes of one direction over `lines` lines (line l at buf + l ls), slots
// k0 .. k0 + np.  Barriers: before the first pass by the caller, after each here.
template <int SIGN, bool DIT>
__device__ __forceinline__ void fx_transform(fx2* buf, int ls, int lines, FxShared& sh, int k0, int M,
                                             const int* __restrict__ nat, const fxw* __restrict__ tw) {
  const int np = sh.np;
  for (int k = 0; k < np; ++k) {
    const int i = DIT ? k : np - 1 - k;
    const FxPass P = sh.p[i];
    const int total = P.units * lines;
    for (int u0 = 0; u0 < total; u0 += blockDim.x) {
      const int u = u0 + threadIdx.x;
      const bool on = u < total;
      int m = 0, line = 0;
      if (on) {
        line = static_cast<int>(fdiv(static_cast<unsigned>(u), P.ulines));
        const int g = fx_shift_of(sh, k0 + k, k0, DIT ? P.bits_dit : P.bits_dif, line);
        int p;
        fx2* base = buf + line * ls + __ldg(&nat[fx_unit_entry(P, u - line * P.units, p)]);
        m = i == 0 ? fx_run_unit<SIGN, DIT, true>(P, base, g, p, M, tw)
                   : fx_run_unit<SIGN, DIT, false>(P, base, g, p, M, tw);
      }
      const int l0 = __shfl_sync(0xffffffffu, line, 0);
      if (__all_sync(0xffffffffu, !on || line == l0)) {
        const int r = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(m)));
        if ((threadIdx.x & 31) == 0 && on) atomicMax(&sh.mag[k0 + k + 1][line], r);
      } else if (on) {
        atomicMax(&sh.mag[k0 + k + 1][line], m);
      }
    }
    __syncthreads();
  }
}

// Exponent change of a line over the passes of one direction.
template <bool DIT>
__device__ __forceinline__ int fx_exponent(const FxShared& sh, int k0, int line) {
  int e = 0;
  for (int k = 0; k < sh.np; ++k) {
    const int i = DIT ? k : sh.np - 1 - k;
    e += 2 * fx_quarters(sh.p[i].shape, i == 0) -
         fx_shift_of(sh, k0 + k, k0, DIT ? sh.p[i].bits_dit : sh.p[i].bits_dif, line);
  }
  return e;
}

constexpr int kFxPlainBits = 59;   // bits of a line without passes (M = 1)
__device__ __forceinline__ int fx_first_bits(const FxShared& sh, bool dit) {
  if (sh.np == 0) return kFxPlainBits;
  return dit ? sh.p[0].bits_dit : sh.p[sh.np - 1].bits_dif;
}
// Biased reference exponent from a largest word (subnormal lines: 1).
__device__ __forceinline__ int fx_ref(int word) {
  const int e = word >> 20;
  return e > 0 ? e : 1;
}

// ---------------------------------------------------------------------------
// column pass: TW (a power of two) neighbouring columns of the flattened
// (outer, inner) range; a thread always handles column threadIdx.x mod TW.
// ---------------------------------------------------------------------------
template <int SIGN>
__device__ __forceinline__ void fx_col_body(const ColArgs& a, const FxPlan& f, int TW, int64_t bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx2* buf = reinterpret_cast<fx2*>(smem_raw);
  __shared__ FxShared sh;
  const int M = f.M;
  const int ls = column_stride(f.ls, TW, sizeof(fx2));
  fx_load_plan(sh, f);
  fx_clear_lines(sh);

  const int t = threadIdx.x & (TW - 1);
  const int i0 = threadIdx.x / TW;                 // TW is a power of two: a shift
  const int di = blockDim.x / TW;
  const int64_t ncols = a.outer * a.inner;
  const int64_t g = bid * TW + t;
  const bool valid = g < ncols;
  const int64_t o = valid ? g / a.inner : 0, jj = valid ? g - o * a.inner : 0;
  const int64_t inner = a.inner;
  const int Lin = SIGN > 0 ? a.Lin : M;
  fx2* line = buf + t * ls;
  grid_wait();
  const double2* __restrict__ in = after_wait(static_cast<const double2*>(a.in) + o * Lin * inner + jj);
  if (a.st != nullptr && a.st->done != RUNNING) return;

  // Largest exponent of the column, then its integers in place (inverse: the
  // digit-reversed positions; forward: natural order).  Columns of up to K
  // entries a thread stay in registers in between; longer ones are read again.
  const bool update = SIGN > 0 && a.pold != nullptr;
  const double2* src = in;
  constexpr int K = 12;
  double2 r[K];
  int mx = 0;
  const double beta = update ? a.st->beta : 0.0;
  const double2* pold = update ? static_cast<const double2*>(a.pold) + o * Lin * inner + jj : in;
  double2* pnew = update ? static_cast<double2*>(a.pnew) + o * Lin * inner + jj : nullptr;
  if (update) src = pnew;   // p = r + beta p_old, written back
  for (int ib = i0; ib < Lin; ib += K * di) {
#pragma unroll
    for (int c = 0; c < K; ++c) {
      const int i = ib + c * di;
      r[c] = make_double2(0.0, 0.0);
      if (valid && i < Lin) r[c] = in[i * inner];
    }
    if (update) {
#pragma unroll
      for (int c = 0; c < K; ++c) {
        const int i = ib + c * di;
        if (valid && i < Lin) {
          const double2 q = pold[i * inner];
          r[c] = make_double2(fma(beta, q.x, r[c].x), fma(beta, q.y, r[c].y));
        }
      }
#pragma unroll
      for (int c = 0; c < K; ++c) {
        const int i = ib + c * di;
        if (valid && i < Lin) pnew[i * inner] = r[c];
      }
    }
#pragma unroll
    for (int c = 0; c < K; ++c) mx = max(mx, max(fx_absword(r[c].x), fx_absword(r[c].y)));
  }
  for (int s = 16; s >= TW; s >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, s));
  __syncthreads();   // plan and cleared slots are in place
  if ((threadIdx.x & 31) < TW) atomicMax(&sh.emax[t], mx);
  __syncthreads();
  const int word = sh.emax[t];
  const bool bad = (word >> 20) == kFxNonFinite;
  const int E = fx_ref(word), bits = fx_first_bits(sh, SIGN > 0);
  const int* __restrict__ perm = f.perm;
  const int* __restrict__ nat = f.nat;
  const int half = (Lin - 1) / 2;

  for (int ib = i0; ib < Lin; ib += K * di) {
    if (Lin > K * di) {
#pragma unroll
      for (int c = 0; c < K; ++c) {
        const int i = ib + c * di;
        r[c] = make_double2(0.0, 0.0);
        if (valid && i < Lin) r[c] = src[i * inner];
      }
    }
#pragma unroll
    for (int c = 0; c < K; ++c) {
      const int i = ib + c * di;
      if (i < Lin) {
        const int k = i - half < 0 ? i - half + M : i - half;
        const int pos = SIGN > 0 ? __ldg(&perm[k]) : __ldg(&nat[i]);
        line[pos] = bad ? fx2{0, 0} : fx2{fx_from_double(r[c].x, E, bits), fx_from_double(r[c].y, E, bits)};
      }
    }
  }
  if (SIGN > 0)
    for (int k = half + 1 + i0; k < M - half; k += di) line[__ldg(&perm[k])] = fx2{0, 0};
  __syncthreads();
  fx_transform<SIGN, (SIGN > 0)>(buf, ls, TW, sh, 0, M, nat, f.tw);

  if (!valid) return;
  FxScale so = fx_scale_of(E - 1022 - bits + fx_exponent<(SIGN > 0)>(sh, 0, t));
  if (SIGN < 0) so.a *= 1.0 / M;
  if (bad) so.a = __longlong_as_double(0x7ff8000000000000LL);
  if (SIGN > 0) {
    double2* out = static_cast<double2*>(a.out) + o * M * inner + jj;
    for (int m = i0; m < M; m += di) {
      const fx2 v = line[__ldg(&nat[m])];
      out[m * inner] = make_double2(fx_to_double(v.x, so), fx_to_double(v.y, so));
    }
  } else {
    const int Lout = a.Lout;
    const int half = (Lout - 1) / 2;
    double2* out = static_cast<double2*>(a.out) + o * Lout * inner + jj;
    for (int i = i0; i < Lout; i += di) {
      const int k = i - half < 0 ? i - half + M : i - half;
      const fx2 v = line[__ldg(&perm[k])];
      out[i * inner] = make_double2(fx_to_double(v.x, so), fx_to_double(v.y, so));
    }
  }
}

// ---------------------------------------------------------------------------
// last-axis pass: NL complex lines (pairs of real lines) of rows_per_cta rows.
// The warps of a CTA are dealt to the lines (several to a line when there are
// fewer lines than warps), so that a warp works on one line at a time.
// ---------------------------------------------------------------------------
struct FxLine {
  int64_t off[2];     // first entry of the two real lines in their fields
  int64_t row[2];
  int field[2];
  int valid;          // bit r: real line r exists
};

__device__ __forceinline__ double2* fx_field(const RowArgs& a, int f) {   // selects: see row_field
  return static_cast<double2*>(f == 0 ? a.t[0] : (f == 1 ? a.t[1] : a.t[2]));
}

// A = (h 2^32 + l) 2^(ex - 1084), the sign in the halves
struct FxMultiplier {
  int h, l, ex;
};
__device__ __forceinline__ FxMultiplier fx_multiplier(double a) {
  long long m;
  int ex;
  fx_split(a, m, ex);
  m >>= 1;
  m = a < 0 ? -m : m;
  return FxMultiplier{fx_hi(m), static_cast<int>(m), ex};
}

template <int MODE>
__device__ __forceinline__ void fx_row_body(const RowArgs& a, const FxPlan& f, int rows_per_cta, int NL, int64_t bid,
                                            int64_t nb) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  fx2* buf = reinterpret_cast<fx2*>(smem_raw);
  __shared__ FxShared sh;
  __shared__ FxLine ld[kFxMaxLines];
  __shared__ double red[32];
  __shared__ bool last;
  const int M = f.M, H = a.H, ls = f.ls;
  const int per_row = a.nfields * a.ncomp;
  const int nrl = rows_per_cta * per_row;
  const int64_t groups = (a.rows + rows_per_cta - 1) / rows_per_cta;
  const int* __restrict__ perm = f.perm;
  const int* __restrict__ nat = f.nat;
  const int lane = threadIdx.x & 31;
  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);
  const int nwarp = blockDim.x >> 5;
  const int segs = nwarp > NL ? nwarp / NL : 1;    // warps per line
  fx_load_plan(sh, f);
  grid_wait();
  if (a.st != nullptr && a.st->done != RUNNING) return;
  double gs[6] = {0, 0, 0, 0, 0, 0};               // ENERGY: upper triangle of F x F, F <= 3

  for (int64_t grp = bid; grp < groups; grp += nb) {
    fx_clear_lines(sh);
    if (threadIdx.x < NL) {
      FxLine d;
      d.valid = 0;
      for (int r = 0; r < 2; ++r) {
        const int rho = 2 * threadIdx.x + r;
        d.row[r] = grp * rows_per_cta + rho / per_row;
        d.field[r] = (rho / a.ncomp) % a.nfields;
        d.off[r] = (rho % a.ncomp) * a.comp_stride + d.row[r] * H;
        if (rho < nrl && d.row[r] < a.rows) d.valid |= 1 << r;
      }
      ld[threadIdx.x] = d;
    }
    __syncthreads();

    // Largest exponent of each line, then Z(k) = X0(k) + i X1(k), Z(-k) = conj
    // X0(k) + i conj X1(k) as integers at their digit-reversed positions, zeros
    // at the frequencies the spectra do not reach.  (The second read comes from
    // L1/L2; held in registers in between the spectra cost spills, 1017 -> 1051
    // us at M = 4374.)
    for (int idx = warp; idx < NL * segs; idx += nwarp) {
      const int j = idx / segs, k0 = (idx - j * segs) * 32 + lane;
      const FxLine d = ld[j];
      const double2* x0 = fx_field(a, d.field[0]) + d.off[0];
      const double2* x1 = fx_field(a, d.field[1]) + d.off[1];
      int mx = 0;
#pragma unroll 4
      for (int k = k0; k < H; k += 32 * segs) {
        double2 A = make_double2(0.0, 0.0), B = make_double2(0.0, 0.0);
        if (d.valid & 1) A = x0[k];
        if (d.valid & 2) B = x1[k];
        mx = max(max(mx, max(fx_absword(A.x), fx_absword(A.y))), max(fx_absword(B.x), fx_absword(B.y)));
      }
      mx = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(mx)));
      if (lane == 0) atomicMax(&sh.emax[j], mx);
    }
    __syncthreads();
    const int bits = fx_first_bits(sh, true) - 1;   // one bit for the sum of two entries
    for (int idx = warp; idx < NL * segs; idx += nwarp) {
      const int j = idx / segs, k0 = (idx - j * segs) * 32 + lane;
      const FxLine d = ld[j];
      const double2* x0 = fx_field(a, d.field[0]) + d.off[0];
      const double2* x1 = fx_field(a, d.field[1]) + d.off[1];
      fx2* line = buf + j * ls;
      const int word = sh.emax[j];
      const int E = fx_ref(word);
      const bool bad = (word >> 20) == kFxNonFinite;
#pragma unroll 2
      for (int k = k0; k < H; k += 32 * segs) {
        double2 A = make_double2(0.0, 0.0), B = make_double2(0.0, 0.0);
        if ((d.valid & 1) && !bad) A = x0[k];
        if ((d.valid & 2) && !bad) B = x1[k];
        const long long ax = fx_from_double(A.x, E, bits), ay = fx_from_double(A.y, E, bits);
        const long long bx = fx_from_double(B.x, E, bits), by = fx_from_double(B.y, E, bits);
        line[__ldg(&perm[k])] = fx2{ax - by, ay + bx};
        if (k > 0) line[__ldg(&perm[M - k])] = fx2{ax + by, bx - ay};
      }
      for (int k = H + k0; k <= M - H; k += 32 * segs) line[__ldg(&perm[k])] = fx2{0, 0};
    }
    __syncthreads();
    fx_transform<+1, true>(buf, ls, NL, sh, 0, M, nat, f.tw);

    if (MODE == ROW_MATVEC) {
      // Multiply by A_M.  The products' largest exponent is found first (from
      // the leading 31 bits of both factors); the products themselves are
      // formed in double (FP64 pipe) at the scale of the line's new reference.
      const double* __restrict__ am = static_cast<const double*>(a.a);
      const int kp = sh.np;                 // slot after the inverse passes
      for (int idx = warp; idx < NL * segs; idx += nwarp) {
        const int j = idx / segs, m0 = (idx - j * segs) * 32 + lane;
        const FxLine d = ld[j];
        const fx2* line = buf + j * ls;
        const double* a0 = am + ((d.valid & 1) ? d.row[0] * M : 0);
        const double* a1 = am + ((d.valid & 2) ? d.row[1] * M : 0);
        int mx = 0;
#pragma unroll 4
        for (int m = m0; m < M; m += 32 * segs) {
          const fx2 u = line[__ldg(&nat[m])];
          const int w0 = static_cast<int>(__double_as_longlong(__ldg(&a0[m])) >> 32) & 0x7fffffff;
          int w1 = w0;
          if (a1 != a0) w1 = static_cast<int>(__double_as_longlong(__ldg(&a1[m])) >> 32) & 0x7fffffff;
          // |u A| < (p + 2) 2^(ex - 990), p = (|u| 2^-32 + 1) (31 leading mantissa bits) 2^-31
          const int c0 = (((w0 & 0xfffff) | 0x100000) << 10) + 1023, c1 = (((w1 & 0xfffff) | 0x100000) << 10) + 1023;
          const int p0 = static_cast<int>((static_cast<long long>(fx_mag(u.x) + 1) * c0) >> 31);
          const int p1 = static_cast<int>((static_cast<long long>(fx_mag(u.y) + 1) * c1) >> 31);
          mx = max(mx, (w0 >> 20) + 32 - __clz(p0 + 2));
          mx = max(mx, (w1 >> 20) + 32 - __clz(p1 + 2));
          if ((w0 >> 20) == kFxNonFinite || (w1 >> 20) == kFxNonFinite) mx = 1 << 20;
        }
        mx = static_cast<int>(__reduce_max_sync(0xffffffffu, static_cast<unsigned>(mx)));
        if (lane == 0) atomicMax(&sh.wmax[j], mx);
      }
      __syncthreads();
      const int wbits = fx_first_bits(sh, false);
      for (int idx = warp; idx < NL * segs; idx += nwarp) {
        const int j = idx / segs, m0 = (idx - j * segs) * 32 + lane;
        const FxLine d = ld[j];
        fx2* line = buf + j * ls;
        const double* a0 = am + ((d.valid & 1) ? d.row[0] * M : 0);
        const double* a1 = am + ((d.valid & 2) ? d.row[1] * M : 0);
        const int s = kp > 0 ? max(62 - fx_bitlen(sh.mag[kp][j]), 0) : 0;
        // u A = (u 2^s C / 2^64) 2^(ex - 1020 - s) with |A| = C 2^(ex - 1084), and
        // |u A| < 2^(wmax - 990): shifted right by wmax - 990 - wbits - (ex - 1020 - s)
        const int c = sh.wmax[j] + 30 - wbits + s;
        auto product = [&](long long u, const FxMultiplier& x) {
          const long long p = fx_mul_add(fx_shl(u, s), x.h, x.l, 0);
          return fx_scale(p, c - x.ex);
        };
        const bool same = a0 == a1;   // both real lines of one row
#pragma unroll 2
        for (int m = m0; m < M; m += 32 * segs) {
          const int pos = __ldg(&nat[m]);
          const fx2 u = line[pos];
          const FxMultiplier x0 = fx_multiplier(__ldg(&a0[m]));
          FxMultiplier x1 = x0;
          if (!same) x1 = fx_multiplier(__ldg(&a1[m]));
          line[pos] = fx2{product(u.x, x0), product(u.y, x1)};
        }
      }
      __syncthreads();
      fx_transform<-1, false>(buf, ls, NL, sh, kp + 1, M, nat, f.tw);

      for (int idx = warp; idx < NL * segs; idx += nwarp) {
        const int j = idx / segs, k0 = (idx - j * segs) * 32 + lane;
        const FxLine d = ld[j];
        double2* x0 = fx_field(a, d.field[0]) + d.off[0];
        double2* x1 = fx_field(a, d.field[1]) + d.off[1];
        const fx2* line = buf + j * ls;
        const int word = sh.emax[j];
        const bool bad = (word >> 20) == kFxNonFinite || sh.wmax[j] >= (1 << 20);
        // exponent of the inverse's output, of the products, of the forward's output; 1/M
        const int eu = fx_ref(word) - 1022 - bits + fx_exponent<true>(sh, 0, j);
        FxScale so = fx_scale_of(eu + sh.wmax[j] - 990 - wbits + fx_exponent<false>(sh, kp + 1, j));
        so.a *= 1.0 / M;
        if (bad) so.a = __longlong_as_double(0x7ff8000000000000LL);
#pragma unroll 2
        for (int k = k0; k < H; k += 32 * segs) {
          const fx2 W = line[__ldg(&perm[k])];
          const fx2 V = line[__ldg(&perm[k == 0 ? 0 : M - k])];
          // X0 = (W + conj V)/2, X1 = (W - conj V)/(2 i)
          if (d.valid & 1)
            x0[k] = make_double2(fx_to_double((W.x + V.x) >> 1, so), fx_to_double((W.y - V.y) >> 1, so));
          if (d.valid & 2)
            x1[k] = make_double2(fx_to_double((W.y + V.y) >> 1, so), fx_to_double((V.x - W.x) >> 1, so));
        }
      }
    } else {
      // real values of the lines (TOREAL: to memory; ENERGY: in place as doubles)
      for (int idx = warp; idx < NL * segs; idx += nwarp) {
        const int j = idx / segs, m0 = (idx - j * segs) * 32 + lane;
        const FxLine d = ld[j];
        fx2* line = buf + j * ls;
        const int word = sh.emax[j];
        const bool bad = (word >> 20) == kFxNonFinite;
        FxScale so = fx_scale_of(fx_ref(word) - 1022 - bits + fx_exponent<true>(sh, 0, j));
        if (bad) so.a = __longlong_as_double(0x7ff8000000000000LL);
        double* out = static_cast<double*>(a.out_real);
        for (int m = m0; m < M; m += 32 * segs) {
          const int pos = __ldg(&nat[m]);
          const fx2 u = line[pos];
          const double2 z = make_double2(fx_to_double(u.x, so), fx_to_double(u.y, so));
          if (MODE == ROW_TOREAL) {
            if (d.valid & 1) out[d.row[0] * M + m] = z.x;
            if (d.valid & 2) out[d.row[1] * M + m] = z.y;
          } else {
            *reinterpret_cast<double2*>(&line[pos]) = z;
          }
        }
      }
      if (MODE == ROW_ENERGY) {   // one row per group, real lines ordered (field, comp)
        __syncthreads();
        const double* __restrict__ am = static_cast<const double*>(a.a);
        const int F = a.nfields, NC = a.ncomp;
        const double* val = reinterpret_cast<const double*>(buf);
        for (int m = threadIdx.x; m < M; m += blockDim.x) {
          const double w = am[ld[0].row[0] * M + m];
          const int pos = __ldg(&nat[m]);
          auto at = [&](int r) { return val[2 * ((r >> 1) * ls + pos) + (r & 1)]; };
          int e = 0;
#pragma unroll
          for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int h2 = i; h2 < 3; ++h2) {
              if (i < F && h2 < F) {
                double s = 0.0;
                for (int c = 0; c < NC; ++c) s = fma(at(i * NC + c), at(h2 * NC + c), s);
                // the entry's place in the upper triangle of F x F
                e = i * F - i * (i - 1) / 2 + (h2 - i);
#pragma unroll
                for (int q = 0; q < 6; ++q)
                  if (q == e) gs[q] = fma(w, s, gs[q]);
              }
            }
        }
      }
    }
    __syncthreads();
  }

  if (MODE == ROW_ENERGY) {
    const int F = a.nfields;
    const int ne = F * (F + 1) / 2;
    for (int e = 0; e < ne; ++e) {
      double mine = 0.0;
#pragma unroll
      for (int q = 0; q < 6; ++q)
        if (q == e) mine = gs[q];
      const double v = block_sum(mine, red);
      if (threadIdx.x == 0) a.partials[bid * 6 + e] = v;
    }
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned int t = atomicAdd(a.ticket, 1u);
      last = (t == nb - 1);
    }
    __syncthreads();
    if (last) {
      __threadfence();
      for (int e = 0; e < ne; ++e) {
        double v = 0.0;
        for (int64_t b = threadIdx.x; b < nb; b += blockDim.x) v += __ldcg(&a.partials[b * 6 + e]);
        v = block_sum(v, red);
        if (threadIdx.x == 0) {
          int ee = 0;
          for (int i = 0; i < F; ++i)
            for (int h2 = i; h2 < F; ++h2, ++ee)
              if (ee == e) {
                a.gram[i * F + h2] = v * a.scale;
                a.gram[h2 * F + i] = v * a.scale;
              }
        }
      }
      if (threadIdx.x == 0) *a.ticket = 0u;
    }
  }
}

// Launch shapes (passes.cu).
int fx_col_tile(int ls, int64_t columns);
int fx_threads(int M, int lines, int ls);
void fx_row_shape(int mode, int nfields, int ncomp, int M, int ls, int64_t rows, int* rows_per_cta, int* NL,
                  int* threads);

// Launchers (fx_col.cu, fx_row.cu).
ghb_status launch_fx_col(int sign, const ColArgs& a, const FxPlan& f, int TW, cudaStream_t s);
ghb_status launch_fx_col_batch(int sign, const ColItem* items, int n, int64_t blocks, size_t smem, int threads,
                               cudaStream_t s);
ghb_status launch_fx_row(int mode, const RowArgs& a, const FxPlan& f, int rows_per_cta, int NL, int threads,
                         cudaStream_t s);
ghb_status launch_fx_row_batch(int mode, const RowItem* items, int n, int64_t blocks, size_t smem, int threads,
                               cudaStream_t s);

}  // namespace ghb
