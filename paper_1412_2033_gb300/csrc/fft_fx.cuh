// Block fixed-point FFT: the FP64 transforms on the integer units.
//
// Why: GB300 issues FP64 at 2 lanes per clock and SM, 1/64 of its FP32 rate
// and 1/32 of its integer rate (measured: FP64 FMA 2.1 lanes/clk/SM, 32x32+64
// bit multiply-add and 64-bit add about 64).  A complex FP64 twiddle product is
// 4 FP64 instructions = 256 scheduler cycles per warp; the same product on
// 64-bit integers is 17 instructions = about 50 cycles, and an addition (two
// instructions) takes 4 cycles instead of 64.  So the double-precision passes hold their data in
// shared memory and registers as 64-bit fixed point with one binary exponent
// per line (block floating point) and convert from and to double where a line
// enters and leaves the CTA.
//
// Numbers.  Entry = v 2^e, v a 64-bit integer per component, e shared by the
// line.  Before every pass the line is shifted so that its largest component
// fills a stated number of bits (about 60); each stage rounds to one unit, that
// is to 2^-60 of the line's largest entry, where double rounds to 2^-53 of each
// entry.  A transform mixes all entries of its line, so in both cases the error
// counts against the line's 2-norm, and the seven extra bits cover the ratio of
// a line's largest entry to its root mean square.
//
// Scaling.  A product with a root of unity w is formed as (v C) / 2^64 with C =
// w 2^62 in two signed 32-bit halves: v w / 4, three 32x32-bit products per
// real product (the low x low one, below one unit, is left out).  Every stage
// with twiddles therefore scales its outputs by 1/4 (entries without a twiddle
// are shifted), which cancels the growth of a radix-3 or radix-4 butterfly, and
// the line's exponent counts the factors of 4.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <cstring>
#include <vector>

#include "fft.cuh"

namespace ghb {

struct alignas(16) fx2 {
  long long x, y;
};

#define FX_HD __host__ __device__ __forceinline__

FX_HD fx2 operator+(fx2 a, fx2 b) { return fx2{a.x + b.x, a.y + b.y}; }
FX_HD fx2 operator-(fx2 a, fx2 b) { return fx2{a.x - b.x, a.y - b.y}; }

// v = fx_hi(v) 2^32 + (int)v, both signed
FX_HD int fx_hi(long long v) { return static_cast<int>(v >> 32) + static_cast<int>(static_cast<unsigned>(v) >> 31); }
// a b + c, as a carry chain over the words of c: one 32 x 32 + 64-bit
// instruction.  (Written as a 64-bit sum the compiler regroups the chains of
// products and spends two more instructions on half of them: a twiddle product
// then takes 31 instructions instead of 17.)
FX_HD long long fx_wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  unsigned lo;
  int hi;
  asm("{\n\t.reg .u32 l, h;\n\tmov.b64 {l, h}, %4;\n\tmad.lo.cc.u32 %0, %2, %3, l;\n\tmadc.hi.s32 %1, %2, %3, h;\n\t}"
      : "=r"(lo), "=r"(hi)
      : "r"(a), "r"(b), "l"(c));
  return static_cast<long long>((static_cast<unsigned long long>(static_cast<unsigned>(hi)) << 32) | lo);
#else
  return static_cast<long long>(a) * b + c;
#endif
}
constexpr long long kFxHalf = 1LL << 31;

// a + v C / 2^64, C = ch 2^32 + cl (|C| <= 2^62, |v| < 2^63), error below one unit
FX_HD long long fx_mul_add(long long v, int ch, int cl, long long a) {
  const int vl = static_cast<int>(v), vh = fx_hi(v);
  const long long cross = fx_wide(vh, cl, fx_wide(vl, ch, kFxHalf));
  return fx_wide(vh, ch, a + (cross >> 32));
}

// a w / 4 (SIGN = -1) or a conj(w) / 4 (SIGN = +1), w in the forward
// convention, |a| <= 2^62.8 (the cross sums stay below 2^63: |ch| + |sh| <=
// sqrt(2) 2^30 against the low halves, |ah| + |bh| <= sqrt(2) |a| 2^-32 against
// the roots' low halves).
template <int SIGN>
FX_HD fx2 fx_cmul4(fx2 a, fxw w) {
  const int sh = SIGN < 0 ? w.sh : -w.sh, sl = SIGN < 0 ? w.sl : -w.sl;
  const int nh = -sh, nl = -sl;
  const int al = static_cast<int>(a.x), ah = fx_hi(a.x);
  const int bl = static_cast<int>(a.y), bh = fx_hi(a.y);
  long long cr = fx_wide(al, w.ch, kFxHalf);
  cr = fx_wide(ah, w.cl, cr);
  cr = fx_wide(bl, nh, cr);
  cr = fx_wide(bh, nl, cr);
  long long ci = fx_wide(al, sh, kFxHalf);
  ci = fx_wide(ah, sl, ci);
  ci = fx_wide(bl, w.ch, ci);
  ci = fx_wide(bh, w.cl, ci);
  fx2 r;
  r.x = fx_wide(bh, nh, fx_wide(ah, w.ch, cr >> 32));
  r.y = fx_wide(bh, w.ch, fx_wide(ah, sh, ci >> 32));
  return r;
}

FX_HD fx2 fx_quarter(fx2 a) { return fx2{(a.x + 2) >> 2, (a.y + 2) >> 2}; }

// ---------------------------------------------------------------------------
// small DFTs X_k = sum_n x_n exp(SIGN 2 pi i n k / R).  Constants k are held as
// the two halves of k 2^64 (|k| < 1/4); a larger one is written as 1 - k or
// 1/2 + k, which costs an addition.
// ---------------------------------------------------------------------------
template <int SIGN>
FX_HD fx2 fx_rot(fx2 a) {   // i SIGN a
  return SIGN > 0 ? fx2{-a.y, a.x} : fx2{a.y, -a.x};
}
template <int SIGN>
FX_HD void fx_dft2(fx2* v) {
  const fx2 a = v[0], b = v[1];
  v[0] = a + b;
  v[1] = a - b;
}
template <int SIGN>
FX_HD void fx_dft3(fx2* v) {
  constexpr int kh = -575416509, kl = -1033546850;   // sqrt(3)/2 - 1
  const fx2 t1 = v[1] + v[2];
  const fx2 d = v[1] - v[2];
  const fx2 t2 = fx2{v[0].x - (t1.x >> 1), v[0].y - (t1.y >> 1)};
  const fx2 s = fx2{fx_mul_add(d.x, kh, kl, d.x), fx_mul_add(d.y, kh, kl, d.y)};
  v[0] = v[0] + t1;
  const fx2 p = fx2{t2.x - s.y, t2.y + s.x};   // t2 + i s
  const fx2 m = fx2{t2.x + s.y, t2.y - s.x};   // t2 - i s
  v[1] = SIGN > 0 ? p : m;
  v[2] = SIGN > 0 ? m : p;
}
template <int SIGN>
FX_HD void fx_dft4(fx2* v) {
  const fx2 a = v[0] + v[2], b = v[0] - v[2];
  const fx2 c = v[1] + v[3], e = fx_rot<SIGN>(v[1] - v[3]);
  v[0] = a + c;
  v[2] = a - c;
  v[1] = b + e;
  v[3] = b - e;
}
// With a1,2 = x1 + x4, x2 + x3 and b1,2 = x1 - x4, x2 - x3:
//   X1,4 = x0 - (a1 + a2)/4 + (sqrt5/4)(a1 - a2) +- i (s1 b1 + s2 b2),
//   X2,3 = x0 - (a1 + a2)/4 - (sqrt5/4)(a1 - a2) +- i (s2 b1 - s1 b2),
// s1 = sin(2 pi/5) = 1 + k1, s2 = sin(4 pi/5) = 1/2 + k2, sqrt5/4 = 1/2 + k0.
template <int SIGN>
FX_HD void fx_dft5(fx2* v) {
  constexpr int k0h = 253476061, k0l = -1079689717;
  constexpr int k1h = -210210662, k1l = 581434099;
  constexpr int k2h = 377034788, k2l = -1429016722;
  const fx2 a1 = v[1] + v[4], b1 = v[1] - v[4];
  const fx2 a2 = v[2] + v[3], b2 = v[2] - v[3];
  const fx2 s = a1 + a2, d = a1 - a2;
  const fx2 c = fx2{v[0].x - ((s.x + 2) >> 2), v[0].y - ((s.y + 2) >> 2)};
  const fx2 e = fx2{fx_mul_add(d.x, k0h, k0l, d.x >> 1), fx_mul_add(d.y, k0h, k0l, d.y >> 1)};
  const fx2 r1 = c + e, r2 = c - e;
  const fx2 s1b1 = fx2{fx_mul_add(b1.x, k1h, k1l, b1.x), fx_mul_add(b1.y, k1h, k1l, b1.y)};
  const fx2 s1b2 = fx2{fx_mul_add(b2.x, k1h, k1l, b2.x), fx_mul_add(b2.y, k1h, k1l, b2.y)};
  const fx2 s2b1 = fx2{fx_mul_add(b1.x, k2h, k2l, b1.x >> 1), fx_mul_add(b1.y, k2h, k2l, b1.y >> 1)};
  const fx2 s2b2 = fx2{fx_mul_add(b2.x, k2h, k2l, b2.x >> 1), fx_mul_add(b2.y, k2h, k2l, b2.y >> 1)};
  const fx2 i1 = fx_rot<SIGN>(s1b1 + s2b2);
  const fx2 i2 = fx_rot<SIGN>(s2b1 - s1b2);
  v[0] = v[0] + s;
  v[1] = r1 + i1;
  v[4] = r1 - i1;
  v[2] = r2 + i2;
  v[3] = r2 - i2;
}
template <int SIGN, int R>
FX_HD void fx_dft(fx2* v) {
  if constexpr (R == 2) fx_dft2<SIGN>(v);
  else if constexpr (R == 3) fx_dft3<SIGN>(v);
  else if constexpr (R == 4) fx_dft4<SIGN>(v);
  else if constexpr (R == 5) fx_dft5<SIGN>(v);
}

// ---------------------------------------------------------------------------
// conversions.  A line's reference E is the largest biased exponent of its
// components (fx_expo); with `bits` b its integers satisfy |v| < 2^b and
// entry = v 2^(E - 1022 - b).
// ---------------------------------------------------------------------------
FX_HD long long fx_bits(double d) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(d);
#else
  long long b;
  memcpy(&b, &d, 8);
  return b;
#endif
}
FX_HD double fx_double(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}
constexpr int kFxNonFinite = 2047;   // biased exponent of infinities and NaN
FX_HD int fx_absword(double d) { return static_cast<int>(fx_bits(d) >> 32) & 0x7fffffff; }   // orders as |d| does
FX_HD int fx_clz(unsigned v) {
#ifdef __CUDA_ARCH__
  return __clz(static_cast<int>(v));
#else
  return v ? __builtin_clz(v) : 32;
#endif
}

// 2^e for e within the normal range, and what is left of e outside +-1000
FX_HD double fx_pow2(int e) { return fx_double(static_cast<long long>(e + 1023) << 52); }
FX_HD int fx_clamp(int e) { return e < -1000 ? -1000 : (e > 1000 ? 1000 : e); }

// Scaling by 2^e in two exact steps (the second is 1 unless |e| > 1000).
struct FxScale {
  double a, b;
  bool two;
};
FX_HD FxScale fx_scale_of(int e) {
  const int e1 = fx_clamp(e), e2 = fx_clamp(e - e1);
  return FxScale{fx_pow2(e1), fx_pow2(e2), e2 != 0};
}
FX_HD double fx_apply(double d, const FxScale& s) {
  d *= s.a;
  return s.two ? d * s.b : d;
}
// Conversions in integer arithmetic (about 18 instructions in, 22 and a product
// out, per component).  A product and a hardware conversion on the FP64 pipe
// are two instructions but hold that pipe for 128 cycles a warp: measured on
// the M = 4374 passes, forward column 427 us against 332, last axis no gain.

// sign and magnitude of a double: |d| = m 2^(ex - 1085), 2^62 <= m < 2^63 (normal d)
FX_HD void fx_split(double d, long long& m, int& ex) {
  const long long b = fx_bits(d);
  const int e = static_cast<int>(b >> 52) & 0x7ff;
  const long long frac = b & 0xfffffffffffffLL;
  ex = e ? e : 1;
  m = (e ? (frac | 0x10000000000000LL) : frac) << 10;
}
FX_HD long long fx_shl(long long v, int g) {
  return static_cast<long long>(static_cast<unsigned long long>(v) << g);
}
// the integer of d in a line of reference E (E < kFxNonFinite) at b bits, rounded to nearest
FX_HD long long fx_from_double(double d, int E, int b) {
  long long m;
  int ex;
  fx_split(d, m, ex);
  int r = 62 - b + (E - ex);   // one less than the right shift 63 - b + E - ex >= 1
  r = r < 63 ? r : 63;
  const long long v = static_cast<long long>(((static_cast<unsigned long long>(m) >> r) + 1) >> 1);
  const long long s = fx_bits(d) >> 63;
  return (v ^ s) - s;
}
// v scaled, as a double: v rounded to 53 bits, then the scale's product
FX_HD double fx_to_double(long long v, const FxScale& s) {
  const int sign = static_cast<int>(v >> 32) >> 31;
  const long long sx = sign;
  unsigned long long u = static_cast<unsigned long long>((v ^ sx) - sx);
#ifdef __CUDA_ARCH__
  const int z = __clzll(static_cast<long long>(u)) & 63;
#else
  const int z = u ? __builtin_clzll(u) : 0;
#endif
  u <<= z;                                                    // leading bit at 63 (unless v = 0)
  const unsigned long long mant = ((u >> 1) + 0x200) >> 10;   // 53 bits with the leading one
  long long bits = static_cast<long long>(mant) + (static_cast<long long>(1085 - z) << 52);
  bits = u ? bits : 0;
  bits |= static_cast<long long>(sign & static_cast<int>(0x80000000u)) << 32;
  return fx_apply(fx_double(bits), s);
}
// v 2^-r rounded (r > 0) or v 2^-r exactly (r <= 0)
FX_HD long long fx_scale(long long v, int r) {
  if (r <= 0) return fx_shl(v, -r);
  if (r > 62) return 0;
  return (v + (1LL << (r - 1))) >> r;
}

// Magnitude of an integer's high word.
FX_HD int fx_mag(long long v) {
  const int h = static_cast<int>(v >> 32);
  return h ^ (h >> 31);
}
// number of bits that hold every value whose fx_mag is at most m
FX_HD int fx_bitlen(int m) { return 64 - fx_clz(static_cast<unsigned>(m)); }
// running minimum and maximum of high words (one three-operand instruction for both components)
FX_HD void fx_track(fx2 v, int& lo, int& hi) {
  const int a = static_cast<int>(v.x >> 32), b = static_cast<int>(v.y >> 32);
#ifdef __CUDA_ARCH__
  lo = __vimin3_s32(lo, a, b);
  hi = __vimax3_s32(hi, a, b);
#else
  lo = a < lo ? a : lo; lo = b < lo ? b : lo;
  hi = a > hi ? a : hi; hi = b > hi ? b : hi;
#endif
}
FX_HD int fx_tracked(int lo, int hi) { return hi > ~lo ? hi : ~lo; }   // lo <= 0 <= hi

// ---------------------------------------------------------------------------
// passes
// ---------------------------------------------------------------------------
// Host side (plan.cu): the passes (k = 0: these, 1: fft_rt.cuh's) of length M with group sizes <= cap, the
// roots of unity and their fixed-point table.
struct UnitRoot {
  long double c, s;   // cos, sin of 2 pi j / M
};
// (perm_out, nat_out: the tables of FxPlan, left out when null).  Spare positions are
// left out as far as the line then takes at most max_ls positions.
bool group_plan(int k, int M, int cap, FxPlan& f, std::vector<int>* perm_out, std::vector<int>* nat_out,
                int max_ls = 1 << 30);
// The most positions a line of length M may take for every launch that admits M to
// fit a CTA's shared memory, `tile` columns a CTA among them.
int line_limit(int k, int M, int tile);
void unit_roots(int M, std::vector<UnitRoot>& r);
void fx_twiddles(const std::vector<UnitRoot>& roots, std::vector<fxw>& tw);

// factors of 4 that a pass takes out: one per stage with twiddles, one for the
// products inside a generic stage
FX_HD int fx_quarters(int shape, bool first) {
  const int n = shape == FX_GENERIC || (shape >= FX_3_2 && shape <= FX_5_2) ? 2 : 1;
  return first ? n - 1 : n;
}

// One sub-stage on the group's entries v (entry j at base + j lp): radix RHO,
// SIG = product of the radices before it in the pass, RG the group's size.
// Twiddle of entry offset JP < SIG, input/output q: w^(q ts_s (p + JP lp)),
// ts_s = M / (lp SIG RHO).  QUARTERED: the entries q = 0 come scaled already.
template <int SIGN, bool DIT, bool FIRST, int RHO, int SIG, int RG, bool QUARTERED>
FX_HD void fx_substage(fx2* v, int p, int lp, int ts, const fxw* __restrict__ tw) {
#pragma unroll
  for (int JP = 0; JP < SIG; ++JP) {
    const bool plain = FIRST && SIG == 1;        // no twiddles at all: no scaling
    const bool unit = FIRST && JP == 0;          // all twiddles are 1
    fxw w[RHO];
    if (!plain && !unit) {
      const int b = ts * (p + JP * lp);
#pragma unroll
      for (int q = 1; q < RHO; ++q) {
#ifdef __CUDA_ARCH__
        const int4 t = __ldg(reinterpret_cast<const int4*>(tw) + q * b);
        w[q] = fxw{t.x, t.y, t.z, t.w};
#else
        w[q] = tw[q * b];
#endif
      }
    }
#pragma unroll
    for (int jb = 0; jb < RG / (SIG * RHO); ++jb) {
      fx2 e[RHO];
#pragma unroll
      for (int q = 0; q < RHO; ++q) e[q] = v[jb * SIG * RHO + JP + q * SIG];
      if (DIT && !plain) {
        if (!QUARTERED) e[0] = fx_quarter(e[0]);
#pragma unroll
        for (int q = 1; q < RHO; ++q) e[q] = unit ? fx_quarter(e[q]) : fx_cmul4<SIGN>(e[q], w[q]);
      }
      fx_dft<SIGN, RHO>(e);
      if (!DIT && !plain) {
        e[0] = fx_quarter(e[0]);
#pragma unroll
        for (int q = 1; q < RHO; ++q) e[q] = unit ? fx_quarter(e[q]) : fx_cmul4<SIGN>(e[q], w[q]);
      }
#pragma unroll
      for (int q = 0; q < RHO; ++q) v[jb * SIG * RHO + JP + q * SIG] = e[q];
    }
  }
}

// One group of a pass: entries at base[j step], normalised by the shift g (left
// if g >= 0), transformed in registers and written back; returns the largest
// fx_mag of the outputs.
template <int SIGN, bool DIT, bool FIRST, int RA, int RB>
FX_HD int fx_group(fx2* base, int step, int g, int p, int lp, int ts, const fxw* __restrict__ tw) {
  constexpr int RG = RA * RB;
  fx2 v[RG];
  // the first stage's entries without a twiddle take its factor 1/4 here
  constexpr bool QUARTERED = DIT && !FIRST;
#pragma unroll
  for (int j = 0; j < RG; ++j) v[j] = base[j * step];
  if (g >= 0) {
#pragma unroll
    for (int j = 0; j < RG; ++j) {
      if (QUARTERED && j % RA == 0) continue;
      v[j] = fx2{static_cast<long long>(static_cast<unsigned long long>(v[j].x) << g),
                 static_cast<long long>(static_cast<unsigned long long>(v[j].y) << g)};
    }
  } else {
    const int r = -g;
    const long long half = 1LL << (r - 1);
#pragma unroll
    for (int j = 0; j < RG; ++j) {
      if (QUARTERED && j % RA == 0) continue;
      v[j] = fx2{(v[j].x + half) >> r, (v[j].y + half) >> r};
    }
  }
  if (QUARTERED) {
    if (g >= 2) {
#pragma unroll
      for (int j = 0; j < RG; j += RA)
        v[j] = fx2{static_cast<long long>(static_cast<unsigned long long>(v[j].x) << (g - 2)),
                   static_cast<long long>(static_cast<unsigned long long>(v[j].y) << (g - 2))};
    } else {
      const int r = 2 - g;
      const long long half = 1LL << (r - 1);
#pragma unroll
      for (int j = 0; j < RG; j += RA) v[j] = fx2{(v[j].x + half) >> r, (v[j].y + half) >> r};
    }
  }
  // ts = M / (lp RG): the sub-stages' steps are ts RB (radix RA) and ts (radix RB)
  if (DIT) {
    fx_substage<SIGN, DIT, FIRST, RA, 1, RG, QUARTERED>(v, p, lp, ts * RB, tw);
    if constexpr (RB > 1) fx_substage<SIGN, DIT, FIRST, RB, RA, RG, false>(v, p, lp, ts, tw);
  } else {
    if constexpr (RB > 1) fx_substage<SIGN, DIT, FIRST, RB, RA, RG, false>(v, p, lp, ts, tw);
    fx_substage<SIGN, DIT, FIRST, RA, 1, RG, false>(v, p, lp, ts * RB, tw);
  }
  int lo = 0, hi = 0;
#pragma unroll
  for (int j = 0; j < RG; ++j) {
    fx_track(v[j], lo, hi);
    base[j * step] = v[j];
  }
  return fx_tracked(lo, hi);
}

// One stage of a prime radix R <= kMaxGenericRadix by the definition (O(R^2)),
// its R-th roots from the length-M table (MR = M / R).
template <int SIGN, bool DIT>
FX_HD int fx_group_generic(fx2* base, int step, int g, int p, int R, int ts, int MR, bool first,
                           const fxw* __restrict__ tw) {
  fx2 v[kMaxGenericRadix], o[kMaxGenericRadix];
  const int r = g < 0 ? -g : 0, l = g < 0 ? 0 : g;
  const long long half = r > 0 ? 1LL << (r - 1) : 0;
  for (int q = 0; q < R; ++q) {
    const fx2 t = base[q * step];
    v[q] = fx2{static_cast<long long>(static_cast<unsigned long long>((t.x + half) >> r) << l),
               static_cast<long long>(static_cast<unsigned long long>((t.y + half) >> r) << l)};
    if (DIT && !first) v[q] = fx_cmul4<SIGN>(v[q], tw[q * p * ts]);
  }
  for (int k = 0; k < R; ++k) {   // scaled by 1/4 (the products with the roots)
    fx2 acc = fx_quarter(v[0]);
    int e = 0;
    for (int n = 1; n < R; ++n) {
      e += k;
      if (e >= R) e -= R;
      acc = acc + fx_cmul4<SIGN>(v[n], tw[e * MR]);
    }
    o[k] = acc;
  }
  int lo = 0, hi = 0;
  for (int q = 0; q < R; ++q) {
    fx2 t = o[q];
    if (!DIT && !first) t = fx_cmul4<SIGN>(t, tw[q * p * ts]);
    fx_track(t, lo, hi);
    base[q * step] = t;
  }
  return fx_tracked(lo, hi);
}

// First entry of unit u of a pass and its offset p < lp.
FX_HD int fx_unit_entry(const FxPass& P, int u, int& p) {
#ifdef __CUDA_ARCH__
  const int b = static_cast<int>(fdiv(static_cast<unsigned>(u), P.ulp));
#else
  const int b = u / P.lp;
#endif
  p = u - b * P.lp;
  return b * (P.lp * P.R) + p;
}

template <int SIGN, bool DIT, bool FIRST>
FX_HD int fx_run_unit(const FxPass& P, fx2* base, int g, int p, int M, const fxw* __restrict__ tw) {
  switch (P.shape) {
    case FX_2: return fx_group<SIGN, DIT, FIRST, 2, 1>(base, P.step, g, p, P.lp, P.ts, tw);
    case FX_3: return fx_group<SIGN, DIT, FIRST, 3, 1>(base, P.step, g, p, P.lp, P.ts, tw);
    case FX_4: return fx_group<SIGN, DIT, FIRST, 4, 1>(base, P.step, g, p, P.lp, P.ts, tw);
    case FX_5: return fx_group<SIGN, DIT, FIRST, 5, 1>(base, P.step, g, p, P.lp, P.ts, tw);
    case FX_3_2: return fx_group<SIGN, DIT, FIRST, 3, 2>(base, P.step, g, p, P.lp, P.ts, tw);
    case FX_4_2: return fx_group<SIGN, DIT, FIRST, 4, 2>(base, P.step, g, p, P.lp, P.ts, tw);
    case FX_3_3: return fx_group<SIGN, DIT, FIRST, 3, 3>(base, P.step, g, p, P.lp, P.ts, tw);
    case FX_5_2: return fx_group<SIGN, DIT, FIRST, 5, 2>(base, P.step, g, p, P.lp, P.ts, tw);
    default: return fx_group_generic<SIGN, DIT>(base, P.step, g, p, P.R, P.ts, M / P.R, FIRST, tw);
  }
}

}  // namespace ghb
