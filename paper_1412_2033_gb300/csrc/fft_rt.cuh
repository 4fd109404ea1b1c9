// FP32 shared-memory FFT for run-time plans: the stages of fft.cuh in passes of up
// to 16 entries a thread, read from a source and handed to a sink where a line
// enters and leaves the CTA.
//
// Strides, unit counts and twiddle steps come from the plan, but a group's
// position is one table look-up (nat, perm) and its entries are evenly spaced,
// so the index work is a few instructions per group.  Large groups matter more
// than registers here: the passes of a short line are bound by latency (loads,
// barriers), and a group of 16 entries has that many loads in flight.
//
// Bound by latency and instruction fetch (at 24 warps an SM the largest stall is
// "no instruction" and 45 % of the cycles issue; 32 warps at 64 registers where a
// launch has work for them, see kRtManyThreads).  Measured against the scalar
// run-time engine this replaces (groups of up to 32 by nested dispatch, padded
// index per entry, a copy into and out of shared memory around every transform):
// N = 1023, M = 2048 last axis 57 -> 41 us, axis 1 52 / 42 -> 20 / 18, operator 154.5
// -> 85 us; 64 mixed microstructures of N = 31 .. 255 468 -> 333 ms.
//
// Pairs of lines in packed arithmetic (fma / add / mul .f32x2, both lines in one
// 16-byte entry) were measured and not kept: the packed forms run at the scalar
// rate per float (65 lanes/clk/SM of two), groups of nine pairs took 0.198
// SM-cycles per point and pass of two stages against 0.305 of three for scalar
// groups of 27, and the column pass at M = 4374 98 us against 64.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>
#include <type_traits>

#include "fft_ct.cuh"

namespace ghb {

// ---------------------------------------------------------------------------
// passes.  A group's entries come from shared memory or from a source src(q, n)
// (line q, natural index n) and go to shared memory or to a sink snk(q, n, v).
// Indices: digit-reversed side (inverse input, forward output; the first pass,
// unit r): n = r + (M / RG) rev(j), rev(d1 + RA d2) = d1 RB + d2; natural side
// (inverse output, forward input; the last pass): n = p + j lp.
// ---------------------------------------------------------------------------
struct RtMem {};   // "in shared memory"

struct RtUnit {
  float2* base;       // position of entry 0
  int q;          // line
  int p;          // offset of entry 0 (0 in the first pass)
  int r;          // first pass: natural index of entry 0
};

// Natural-side weight of the group's entry j = d1 + RA d2.
template <int RA, int RB>
__host__ __device__ constexpr int rt_rev(int j) {
  return (j % RA) * RB + j / RA;
}

// All stages of a group on its entries v: ts = M / (lp RA RB); the first
// pass (p = 0) has compile-time roots only.
template <int SIGN, bool DIT, bool FIRST, int RHO, int SIG, int RG>
__device__ __forceinline__ void rt_stage(float2* v, int p, int ts, const float2* __restrict__ tw) {
  if constexpr (FIRST) substage_const<SIGN, DIT, RHO, SIG, RG, 0>(v);
  else substage_jp<SIGN, DIT, RHO, SIG, RG, 0>(v, __ldg(&tw[p * ts]));
}
template <int SIGN, bool DIT, bool FIRST, int RA, int RB>
__device__ __forceinline__ void rt_stages(float2* v, int p, int ts, const float2* __restrict__ tw) {
  constexpr int RG = RA * RB;
  if constexpr (DIT) {
    rt_stage<SIGN, DIT, FIRST, RA, 1, RG>(v, p, ts * RB, tw);
    if constexpr (RB > 1) rt_stage<SIGN, DIT, FIRST, RB, RA, RG>(v, p, ts, tw);
  } else {
    if constexpr (RB > 1) rt_stage<SIGN, DIT, FIRST, RB, RA, RG>(v, p, ts, tw);
    rt_stage<SIGN, DIT, FIRST, RA, 1, RG>(v, p, ts * RB, tw);
  }
}

template <typename F>
constexpr bool rt_is_mem = std::is_same<F, RtMem>::value;
// sources with kUpdate = true also get store(q, n, v) once a unit's entries are all read
template <typename S, typename = void>
struct rt_updates : std::false_type {};
template <typename S>
struct rt_updates<S, std::void_t<decltype(S::kUpdate)>> : std::integral_constant<bool, S::kUpdate> {};

template <int SIGN, bool DIT, bool FIRST, int RA, int RB, typename Src, typename Snk>
__device__ __forceinline__ void rt_group(const FxPass& P, const RtUnit& u, const float2* __restrict__ tw, const Src& src,
                                         const Snk& snk) {
  constexpr int RG = RA * RB;
  float2 v[RG];
  auto rev = [&](int j) { return u.r + P.units * rt_rev<RA, RB>(j); };   // M / RG = units
  auto nat = [&](int j) { return u.p + j * P.lp; };
#pragma unroll
  for (int j = 0; j < RG; ++j) {
    if constexpr (!rt_is_mem<Src>) v[j] = src(u.q, DIT ? rev(j) : nat(j));
    else v[j] = u.base[j * P.step];
  }
  if constexpr (rt_updates<Src>::value) {
#pragma unroll
    for (int j = 0; j < RG; ++j) src.store(u.q, rev(j), v[j]);
  }
  rt_stages<SIGN, DIT, FIRST, RA, RB>(v, u.p, P.ts, tw);
#pragma unroll
  for (int j = 0; j < RG; ++j) {
    if constexpr (!rt_is_mem<Snk>) snk(u.q, DIT ? nat(j) : rev(j), v[j]);
    else u.base[j * P.step] = v[j];
  }
}

// The last inverse pass, a pointwise product mul(q, m, v) and the first forward
// pass act on the same entries p + j lp of the natural order: one thread does
// the three in registers (plans of two passes or more).
template <int RA, int RB, typename Mul>
__device__ __forceinline__ void rt_fused(const FxPass& P, const RtUnit& u, const float2* __restrict__ tw, const Mul& mul) {
  constexpr int RG = RA * RB;
  float2 v[RG];
#pragma unroll
  for (int j = 0; j < RG; ++j) v[j] = u.base[j * P.step];
  rt_stages<+1, true, false, RA, RB>(v, u.p, P.ts, tw);
#pragma unroll
  for (int j = 0; j < RG; ++j) v[j] = mul(u.q, u.p + j * P.lp, v[j]);
  rt_stages<-1, false, false, RA, RB>(v, u.p, P.ts, tw);
#pragma unroll
  for (int j = 0; j < RG; ++j) u.base[j * P.step] = v[j];
}

// One stage of a prime radix R <= kMaxGenericRadix by the definition (O(R^2)), its R-th
// roots from the length-M table.  With a_n = x_n + x_{R-n}, b_n = x_n - x_{R-n} and w^n
// = c_n + i s_n, X_k and X_{R-k} are x_0 + sum a_n c_{kn} +- i sum b_n s_{kn}, n = 1 ..
// (R-1)/2: a quarter of the products of the plain sum, and of the table's loads.
// Measured, one operator application against the plain sum: M = 2002 (2 7 11 13) 565 ->
// 420 us, M = 242 (2 11 11) 82 -> 67, M = 62 (2 31) 128 -> 76, d = 3 M = 130 236 -> 186; the
// scalar run-time engine before this file took 498, 74, 122 and 539.
template <int SIGN, bool DIT>
__device__ __noinline__ void rt_generic_stage(float2* v, int p, int R, int ts, int MR, const float2* __restrict__ tw) {
  float2 o[kMaxGenericRadix];
  const int h = R / 2;
  if (DIT)
    for (int q = 1; q < R; ++q) v[q] = twmul<SIGN>(v[q], __ldg(&tw[q * p * ts]));
  const float2 x0 = v[0];
  float2 sum = x0;
  for (int n = 1; n <= h; ++n) {
    const float2 a = v[n] + v[R - n], b = v[n] - v[R - n];
    v[n] = a;
    v[R - n] = b;
    sum = sum + a;
  }
  o[0] = sum;
  for (int k = 1; k <= h; ++k) {
    float2 c = x0, s = make_float2(0.0f, 0.0f);
    int e = 0;
    for (int n = 1; n <= h; ++n) {
      e += k;
      if (e >= R) e -= R;
      const float2 w = __ldg(&tw[e * MR]);   // (cos, -sin)
      const float2 a = v[n], b = v[R - n];
      c = make_float2(fmaf(w.x, a.x, c.x), fmaf(w.x, a.y, c.y));
      s = make_float2(fmaf(w.y, b.x, s.x), fmaf(w.y, b.y, s.y));
    }
    const float2 r = rot<-SIGN>(s);   // i SIGN sum b sin
    o[k] = c + r;
    o[R - k] = c - r;
  }
  for (int q = 0; q < R; ++q) v[q] = (!DIT && q > 0) ? twmul<SIGN>(o[q], __ldg(&tw[q * p * ts])) : o[q];
}
template <int SIGN, bool DIT, typename Src, typename Snk>
__device__ __forceinline__ void rt_group_generic(const FxPass& P, const RtUnit& u, int M, const float2* __restrict__ tw,
                                                 const Src& src, const Snk& snk) {
  float2 v[kMaxGenericRadix];
  auto rev = [&](int j) { return u.r + P.units * j; };
  auto nat = [&](int j) { return u.p + j * P.lp; };
  for (int j = 0; j < P.R; ++j) {
    if constexpr (!rt_is_mem<Src>) {
      v[j] = src(u.q, DIT ? rev(j) : nat(j));
      if constexpr (rt_updates<Src>::value) src.store(u.q, rev(j), v[j]);
    } else {
      v[j] = u.base[j * P.step];
    }
  }
  rt_generic_stage<SIGN, DIT>(v, u.p, P.R, P.ts, M / P.R, tw);
  for (int j = 0; j < P.R; ++j) {
    if constexpr (!rt_is_mem<Snk>) snk(u.q, DIT ? nat(j) : rev(j), v[j]);
    else u.base[j * P.step] = v[j];
  }
}

template <int SIGN, bool DIT, bool FIRST, typename Src, typename Snk>
__device__ __forceinline__ void rt_run_unit(const FxPass& P, const RtUnit& u, int M, const float2* __restrict__ tw,
                                            const Src& src, const Snk& snk) {
  switch (P.shape) {
    case RT_2: rt_group<SIGN, DIT, FIRST, 2, 1>(P, u, tw, src, snk); break;
    case RT_3: rt_group<SIGN, DIT, FIRST, 3, 1>(P, u, tw, src, snk); break;
    case RT_4: rt_group<SIGN, DIT, FIRST, 4, 1>(P, u, tw, src, snk); break;
    case RT_5: rt_group<SIGN, DIT, FIRST, 5, 1>(P, u, tw, src, snk); break;
    case RT_3_2: rt_group<SIGN, DIT, FIRST, 3, 2>(P, u, tw, src, snk); break;
    case RT_4_2: rt_group<SIGN, DIT, FIRST, 4, 2>(P, u, tw, src, snk); break;
    case RT_3_3: rt_group<SIGN, DIT, FIRST, 3, 3>(P, u, tw, src, snk); break;
    case RT_5_2: rt_group<SIGN, DIT, FIRST, 5, 2>(P, u, tw, src, snk); break;
    case RT_3_4: rt_group<SIGN, DIT, FIRST, 3, 4>(P, u, tw, src, snk); break;
    case RT_5_3: rt_group<SIGN, DIT, FIRST, 5, 3>(P, u, tw, src, snk); break;
    case RT_4_4: rt_group<SIGN, DIT, FIRST, 4, 4>(P, u, tw, src, snk); break;
    default: rt_group_generic<SIGN, DIT>(P, u, M, tw, src, snk); break;
  }
}

template <typename Mul>
__device__ __forceinline__ void rt_run_fused(const FxPass& P, const RtUnit& u, int M, const float2* __restrict__ tw,
                                             const Mul& mul) {
  switch (P.shape) {
    case RT_2: rt_fused<2, 1>(P, u, tw, mul); break;
    case RT_3: rt_fused<3, 1>(P, u, tw, mul); break;
    case RT_4: rt_fused<4, 1>(P, u, tw, mul); break;
    case RT_5: rt_fused<5, 1>(P, u, tw, mul); break;
    case RT_3_2: rt_fused<3, 2>(P, u, tw, mul); break;
    case RT_4_2: rt_fused<4, 2>(P, u, tw, mul); break;
    case RT_3_3: rt_fused<3, 3>(P, u, tw, mul); break;
    case RT_5_2: rt_fused<5, 2>(P, u, tw, mul); break;
    case RT_3_4: rt_fused<3, 4>(P, u, tw, mul); break;
    case RT_5_3: rt_fused<5, 3>(P, u, tw, mul); break;
    case RT_4_4: rt_fused<4, 4>(P, u, tw, mul); break;
    default: {
      rt_group_generic<+1, true>(P, u, M, tw, RtMem(), RtMem());
      for (int j = 0; j < P.R; ++j) u.base[j * P.step] = mul(u.q, u.p + j * P.lp, u.base[j * P.step]);
      rt_group_generic<-1, false>(P, u, M, tw, RtMem(), RtMem());
      break;
    }
  }
}

}  // namespace ghb
