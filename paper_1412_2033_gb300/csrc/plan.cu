// FFT plans: factorisation of M, digit-reversal permutation, twiddle tables.
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "fft_ct.cuh"
#include "fft_fx.cuh"
#include "ghb_internal.cuh"

namespace ghb {

namespace {

bool factor(int M, std::vector<int>& radices) {
  radices.clear();
  int m = M;
  while (m % 4 == 0) { radices.push_back(4); m /= 4; }
  while (m % 2 == 0) { radices.push_back(2); m /= 2; }
  while (m % 3 == 0) { radices.push_back(3); m /= 3; }
  while (m % 5 == 0) { radices.push_back(5); m /= 5; }
  for (int p = 7; p <= kMaxGenericRadix && m > 1; p += 2) {
    while (m % p == 0) { radices.push_back(p); m /= p; }
  }
  return m == 1 && static_cast<int>(radices.size()) <= kMaxStages;
}

struct Shape {
  int id;
  int r[3];
};

// Pass shapes in DIT radix order (see PassShape); longest first.
const Shape kShapes[] = {
    {SH_2_3_3, {2, 3, 3}}, {SH_3_3_3, {3, 3, 3}}, {SH_4_2_3, {4, 2, 3}}, {SH_2_3_5, {2, 3, 5}},
    {SH_4_4_2, {4, 4, 2}}, {SH_2_3, {2, 3, 0}},   {SH_3_3, {3, 3, 0}},   {SH_2_5, {2, 5, 0}},
    {SH_4_3, {4, 3, 0}},   {SH_3_5, {3, 5, 0}},   {SH_4_4, {4, 4, 0}},   {SH_4_5, {4, 5, 0}},
    {SH_5_5, {5, 5, 0}},   {SH_4_2, {4, 2, 0}},   {SH_2, {2, 0, 0}},     {SH_3, {3, 0, 0}},
    {SH_4, {4, 0, 0}},     {SH_5, {5, 0, 0}},
};

}  // namespace

// Group consecutive stages into passes: at each stage take the first (longest)
// shape that matches the next radices with radix product <= maxprod.
void group_passes(FftPlan& p, int maxprod) {
  int t = 0, np = 0;
  while (t < p.nst) {
    int best = -1, blen = 0;
    for (const Shape& sh : kShapes) {
      int len = 0;
      while (len < 3 && sh.r[len] != 0) ++len;
      if (t + len > p.nst) continue;
      int prod = 1;
      for (int q = 0; q < len; ++q) prod *= sh.r[q];
      if (prod > maxprod) continue;
      bool ok = true;
      for (int k = 0; k < len; ++k) ok = ok && (p.R[t + k] == sh.r[k]);
      if (ok && len > blen) {
        best = sh.id;
        blen = len;
      }
    }
    int prod = 1;
    if (best < 0) {
      best = SH_GENERIC;
      blen = 1;
    }
    for (int k = 0; k < blen; ++k) prod *= p.R[t + k];
    p.pshape[np] = best;
    p.pR[np] = prod;
    p.pLp[np] = p.Lp[t];
    p.pdiv[np] = make_fastdiv(static_cast<unsigned>(p.Lp[t]));
    ++np;
    t += blen;
  }
  p.npass = np;
  for (int i = np; i < kMaxPasses; ++i) {
    p.pshape[i] = SH_2;
    p.pR[i] = 1;
    p.pLp[i] = 1;
    p.pdiv[i] = make_fastdiv(1);
  }
}

namespace {

struct FxShapeDef {
  int id, ra, rb;
};
const FxShapeDef kFxShapes[] = {{FX_5_2, 5, 2}, {FX_3_3, 3, 3}, {FX_4_2, 4, 2}, {FX_3_2, 3, 2},
                                {FX_5, 5, 1},   {FX_4, 4, 1},   {FX_3, 3, 1},   {FX_2, 2, 1}};

// The fewest passes of product <= cap that multiply to 2^a 3^b 5^c (the first
// found: large shapes first).
bool fx_cover(int a, int b, int c, int cap, int left, std::vector<int>& out) {
  if (a == 0 && b == 0 && c == 0) return true;
  if (left == 0) return false;
  for (int i = 0; i < static_cast<int>(sizeof(kFxShapes) / sizeof(kFxShapes[0])); ++i) {
    const FxShapeDef& s = kFxShapes[i];
    if (s.ra * s.rb > cap) continue;
    if (!out.empty() && i < out.back()) continue;   // in list order: each multiset once
    int da = 0, db = 0, dc = 0;
    for (int r : {s.ra, s.rb}) {
      if (r == 2) da += 1;
      if (r == 4) da += 2;
      if (r == 3) db += 1;
      if (r == 5) dc += 1;
    }
    if (da > a || db > b || dc > c) continue;
    out.push_back(i);
    if (fx_cover(a - da, b - db, c - dc, cap, left - 1, out)) return true;
    out.pop_back();
  }
  return false;
}

}  // namespace

// Passes of the fixed-point transform (fft_fx.cuh): as few as the cap allows,
// odd group sizes first (the first pass's threads then sit at an odd stride),
// primes above 5 last.
bool fx_group_passes(int M, int cap, FxPlan& f, std::vector<int>* perm_out) {
  int a = 0, b = 0, c = 0, m = M;
  while (m % 2 == 0) { ++a; m /= 2; }
  while (m % 3 == 0) { ++b; m /= 3; }
  while (m % 5 == 0) { ++c; m /= 5; }
  std::vector<int> sh;
  bool ok = false;
  for (int n = 0; n <= kFxPasses && !ok; ++n) {
    sh.clear();
    ok = fx_cover(a, b, c, cap < 5 ? 5 : cap, n, sh);
  }
  if (!ok) return false;
  struct P {
    int id, ra, rb;
  };
  std::vector<P> ps;
  for (int i : sh) ps.push_back(P{kFxShapes[i].id, kFxShapes[i].ra, kFxShapes[i].rb});
  std::stable_sort(ps.begin(), ps.end(), [](const P& x, const P& y) {
    const int px = x.ra * x.rb, py = y.ra * y.rb;
    if ((px & 1) != (py & 1)) return (px & 1) > (py & 1);
    return px > py;
  });
  for (int p = 7; p <= kMaxGenericRadix && m > 1; p += 2)
    while (m % p == 0) {
      ps.push_back(P{FX_GENERIC, p, 1});
      m /= p;
    }
  if (m != 1 || static_cast<int>(ps.size()) > kFxPasses) return false;
  f.np = static_cast<int>(ps.size());
  const int first = f.np > 0 ? ps[0].ra * ps[0].rb : 1;
  f.pad = (f.np > 0 && first % 4 == 0 && first >= 8) ? first : 0;   // strides 2, 6, 10: two-way conflicts only
  f.pdiv = make_fastdiv(static_cast<unsigned>(f.pad > 0 ? f.pad : 1));
  f.ls = M + (f.pad > 0 ? M / f.pad : 0);
  int lp = 1;
  std::vector<int> radix;
  for (int i = 0; i < kFxPasses; ++i) {
    FxPass& q = f.p[i];
    q = FxPass{};
    if (i >= f.np) {
      q.ulines = q.ulp = make_fastdiv(1);
      continue;
    }
    const int R = ps[i].ra * ps[i].rb;
    q.shape = ps[i].id;
    q.R = R;
    q.lp = lp;
    q.step = lp + (f.pad > 0 ? lp / f.pad : 0);
    q.block = lp * R + (f.pad > 0 ? lp * R / f.pad : 0);
    q.units = M / R;
    q.ts = M / (lp * R);
    q.ulines = make_fastdiv(static_cast<unsigned>(q.units));
    q.ulp = make_fastdiv(static_cast<unsigned>(lp));
    // A group's values must stay below 2^62 (fx_cmul4): with largest component
    // 2^b before the pass, magnitudes start at 2^(b + 1/2) and grow by at most
    // R / 4 per scaled stage, R where the factor 1/4 comes after the sums
    // (forward) or not at all (the first pass's first stage).
    const double lr = std::log2(static_cast<double>(q.shape == FX_GENERIC ? R : 5));
    if (q.shape == FX_GENERIC) {
      q.bits_dif = static_cast<int>(std::floor(61.5 - (lr - 2)));
      q.bits_dit = i == 0 ? q.bits_dif : static_cast<int>(std::floor(61.5 - std::max(0.0, lr - 4)));
    } else {
      q.bits_dif = 59;
      q.bits_dit = i == 0 ? static_cast<int>(std::floor(61.0 - std::log2(static_cast<double>(ps[i].ra)))) : 61;
    }
    radix.push_back(ps[i].ra);
    if (ps[i].rb > 1) radix.push_back(ps[i].rb);
    lp *= R;
  }
  if (perm_out) {
    std::vector<int>& perm = *perm_out;
    perm.assign(M, 0);
    std::vector<int> q(radix.size());
    for (int n = 0; n < M; ++n) {
      int rem = n;
      for (int t = static_cast<int>(radix.size()) - 1; t >= 0; --t) {
        q[t] = rem % radix[t];
        rem /= radix[t];
      }
      int pos = 0, L = 1;
      for (size_t t = 0; t < radix.size(); ++t) {
        pos += q[t] * L;
        L *= radix[t];
      }
      perm[n] = pos + (f.pad > 0 ? pos / f.pad : 0);
    }
  }
  return true;
}

// cos and sin of 2 pi j / M for j = 0 .. M-1, each evaluated at an angle of the
// first octant (exact integer reduction, so the angle is rounded below 2^-64)
// and every octant from the first.
void unit_roots(int M, std::vector<UnitRoot>& r) {
  const long double two_pi = 6.283185307179586476925286766559005768L;
  r.resize(M);
  for (int j = 0; j < M; ++j) {
    // 8 j = o M + t: octant o, remainder t; odd octants count back from the next axis or diagonal
    const long long o = (8LL * j) / M, t = (8LL * j) % M;
    const long long u = (o & 1) ? M - t : t;             // angle = 2 pi u / (8 M) in [0, pi/4]
    long double c, s;
    if (j > 0 && o == 7) {   // mirror of M - j (first octant)
      c = r[M - j].c;
      s = r[M - j].s;
    } else {
      const long double x = two_pi * static_cast<long double>(u) / (8.0L * static_cast<long double>(M));
      c = std::cos(x);
      s = std::sin(x);
    }
    // octants 0, 7: (c, +-s); 1, 2: x from the y axis; 3, 4: from the -x axis; 5, 6: from the -y axis
    switch (o) {
      case 0: r[j] = {c, s}; break;
      case 1: r[j] = {s, c}; break;
      case 2: r[j] = {-s, c}; break;
      case 3: r[j] = {-c, s}; break;
      case 4: r[j] = {-c, -s}; break;
      case 5: r[j] = {-s, -c}; break;
      case 6: r[j] = {s, -c}; break;
      default: r[j] = {c, -s}; break;
    }
  }
}

// Roots exp(-2 pi i j / M) 2^62 in balanced halves.
void fx_twiddles(const std::vector<UnitRoot>& roots, std::vector<fxw>& tw) {
  const int M = static_cast<int>(roots.size());
  tw.resize(M);
  auto halves = [](long long v, int& h, int& l) {
    h = static_cast<int>((v + 0x80000000LL) >> 32);
    l = static_cast<int>(v - static_cast<long long>(h) * 4294967296LL);
    if (l == INT32_MIN) l = INT32_MIN + 1;   // one unit of 2^-62: negation must not overflow
  };
  for (int j = 0; j < M; ++j) {
    halves(std::llround(roots[j].c * 4611686018427387904.0L), tw[j].ch, tw[j].cl);
    halves(std::llround(-roots[j].s * 4611686018427387904.0L), tw[j].sh, tw[j].sl);
  }
}

bool factorizable(int M) {
  std::vector<int> r;
  return M >= 1 && factor(M, r);
}

// Smallest M >= 2N - 1 with prime factors 2, 3, 5 only (Lemma integ_eval_VM
// allows any M >= 2N - 1; 5-smooth sizes keep every stage a specialised radix).
int auto_M(int N) {
  for (int M = 2 * N - 1;; ++M) {
    int m = M;
    for (int p : {2, 3, 5}) while (m % p == 0) m /= p;
    if (m == 1) return M;
  }
}

ghb_status build_plan_tables(int M, FftPlan& p, PlanTables& t) {
  std::vector<int> radices;
  if (M < 1 || !factor(M, radices)) {
    set_error("unsupported transform length M=" + std::to_string(M) +
              " (prime factors must be <= 31)");
    return GHB_ERR_INVALID;
  }
  p = FftPlan{};
  p.M = M;
  p.nst = static_cast<int>(radices.size());
  int L = 1;
  for (int t = 0; t < p.nst; ++t) {
    p.R[t] = radices[t];
    p.Lp[t] = L;
    L *= radices[t];
  }
  for (int t = p.nst; t < kMaxStages; ++t) { p.R[t] = 1; p.Lp[t] = L; }
  group_passes(p, 32);
  if (!fx_group_passes(M, kFxCap, p.fx, &t.fx_perm)) {
    set_error("internal: no FP64 passes for M=" + std::to_string(M));
    return GHB_ERR_INVALID;
  }

  // perm[n]: write n in mixed radix with the last stage's radix least
  // significant; the position has the digits in stage order, first stage least
  // significant.
  std::vector<int>& perm = t.perm;
  perm.assign(M, 0);
  std::vector<int> q(p.nst > 0 ? p.nst : 1);
  for (int n = 0; n < M; ++n) {
    int rem = n;
    for (int t = p.nst - 1; t >= 0; --t) {
      q[t] = rem % p.R[t];
      rem /= p.R[t];
    }
    int pos = 0;
    for (int t = 0; t < p.nst; ++t) pos += q[t] * p.Lp[t];
    perm[n] = pos;
  }
  std::vector<UnitRoot> roots;
  unit_roots(M, roots);
  fx_twiddles(roots, t.fx_tw);
  std::vector<float2>& tw32 = t.tw32;
  tw32.resize(M);
  for (int j = 0; j < M; ++j)
    tw32[j] = make_float2(static_cast<float>(static_cast<double>(roots[j].c)),
                          static_cast<float>(-static_cast<double>(roots[j].s)));
  return GHB_OK;
}

ghb_status make_plan(int M, PlanHolder& out) {
  ghb_status st = make_plan_untuned(M, out);
  if (st != GHB_OK) return st;
  return apply_tune(M, out);
}

ghb_status set_fx_cap(PlanHolder& out, int cap) {
  FftPlan& p = out.plan;
  FxPlan f = p.fx;
  std::vector<int> perm;
  if (!fx_group_passes(p.M, cap, f, &perm)) {
    set_error("internal: no FP64 passes for M=" + std::to_string(p.M));
    return GHB_ERR_INVALID;
  }
  GHB_CUDA_TRY(cudaMemcpy(out.d_fx_perm, perm.data(), sizeof(int) * p.M, cudaMemcpyHostToDevice));
  GHB_CUDA_TRY(cudaStreamSynchronize(cudaStreamLegacy));   // in place before any stream's kernels read it
  f.perm = out.d_fx_perm;
  f.tw = p.fx.tw;
  p.fx = f;
  out.fx_cap = cap;
  return GHB_OK;
}

ghb_status make_plan_untuned(int M, PlanHolder& out) {
  PlanTables t;
  ghb_status st = build_plan_tables(M, out.plan, t);
  if (st != GHB_OK) return st;
  FftPlan& p = out.plan;
  const std::vector<int>& perm = t.perm;
  const std::vector<float2>& tw32 = t.tw32;
  GHB_CUDA_TRY(cudaMalloc(&out.d_perm, sizeof(int) * M));
  GHB_CUDA_TRY(cudaMalloc(&out.d_fx_perm, sizeof(int) * M));
  GHB_CUDA_TRY(cudaMalloc(&out.d_fx_tw, sizeof(fxw) * M));
  GHB_CUDA_TRY(cudaMalloc(&out.d_tw32, sizeof(float2) * M));
  GHB_CUDA_TRY(cudaMemcpy(out.d_perm, perm.data(), sizeof(int) * M, cudaMemcpyHostToDevice));
  GHB_CUDA_TRY(cudaMemcpy(out.d_fx_perm, t.fx_perm.data(), sizeof(int) * M, cudaMemcpyHostToDevice));
  GHB_CUDA_TRY(cudaMemcpy(out.d_fx_tw, t.fx_tw.data(), sizeof(fxw) * M, cudaMemcpyHostToDevice));
  GHB_CUDA_TRY(cudaMemcpy(out.d_tw32, tw32.data(), sizeof(float2) * M, cudaMemcpyHostToDevice));
  GHB_CUDA_TRY(cudaStreamSynchronize(cudaStreamLegacy));   // pageable copies: in place before other streams read
  if (ct_size(M) && ct_plan(M).ok) {
    std::vector<int> pct(M);
    ct_perm(M, pct.data());
    GHB_CUDA_TRY(cudaMalloc(&out.d_perm_ct, sizeof(int) * M));
    GHB_CUDA_TRY(cudaMemcpy(out.d_perm_ct, pct.data(), sizeof(int) * M, cudaMemcpyHostToDevice));
  }
  p.perm = out.d_perm;
  p.perm_ct = out.d_perm_ct;
  p.ct_col = p.ct_row = (out.d_perm_ct != nullptr) ? 1 : 0;
  p.fx.perm = out.d_fx_perm;
  p.fx.tw = out.d_fx_tw;
  out.fx_cap = kFxCap;
  p.tw32 = out.d_tw32;
  return GHB_OK;
}

void free_plan(PlanHolder& p) {
  if (p.d_perm) cudaFree(p.d_perm);
  if (p.d_perm_ct) cudaFree(p.d_perm_ct);
  if (p.d_fx_perm) cudaFree(p.d_fx_perm);
  if (p.d_fx_tw) cudaFree(p.d_fx_tw);
  if (p.d_tw32) cudaFree(p.d_tw32);
  p = PlanHolder{};
}

}  // namespace ghb
