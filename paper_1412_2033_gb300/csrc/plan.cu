// FFT plans: factorisation of M, digit-reversal permutation, twiddle tables.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
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

struct GroupShape {
  int id, r[2];
};
const GroupShape kFxShapes[] = {{FX_5_2, {5, 2}}, {FX_3_3, {3, 3}}, {FX_4_2, {4, 2}}, {FX_3_2, {3, 2}},
                                {FX_5, {5, 1}},   {FX_4, {4, 1}},   {FX_3, {3, 1}},   {FX_2, {2, 1}}};
const GroupShape kRtShapes[] = {{RT_4_4, {4, 4}}, {RT_5_3, {5, 3}}, {RT_3_4, {3, 4}}, {RT_5_2, {5, 2}},
                                {RT_3_3, {3, 3}}, {RT_4_2, {4, 2}}, {RT_3_2, {3, 2}}, {RT_5, {5, 1}},
                                {RT_4, {4, 1}},   {RT_3, {3, 1}},   {RT_2, {2, 1}}};

// The groups of product <= cap, `left` of them in list order from `from`, that
// multiply to 2^a 3^b 5^c with the least sum of sizes (balanced: a pass's threads
// go with the number of its groups).
struct Cover {
  const GroupShape* shapes;
  int count, cap;
  std::vector<int> now, best;
  int best_sum = INT_MAX;
  void search(int a, int b, int c, int from, int left, int sum) {
    if (a == 0 && b == 0 && c == 0) {
      if (left == 0 && sum < best_sum) {
        best_sum = sum;
        best = now;
      }
      return;
    }
    if (left == 0) return;
    for (int i = from; i < count; ++i) {
      const int* r = shapes[i].r;
      const int size = r[0] * r[1];
      if (size > cap) continue;
      int d[3] = {0, 0, 0};   // exponents of 2, 3, 5
      for (int k = 0; k < 2; ++k) {
        d[0] += r[k] == 2 ? 1 : (r[k] == 4 ? 2 : 0);
        d[1] += r[k] == 3;
        d[2] += r[k] == 5;
      }
      if (d[0] > a || d[1] > b || d[2] > c) continue;
      now.push_back(i);
      search(a - d[0], b - d[1], c - d[2], i, left - 1, sum + size);
      now.pop_back();
    }
  }
};

}  // namespace

// Passes of a run-time transform (k = 0: fft_fx.cuh, 1: fft_rt.cuh): as few as the
// cap allows, odd group sizes first (the first pass's threads then sit at an odd
// stride), primes above 5 last.
bool group_plan(int k, int M, int cap, FxPlan& f, std::vector<int>* perm_out, std::vector<int>* nat_out, int max_ls) {
  f.M = M;
  int a = 0, b = 0, c = 0, m = M;
  while (m % 2 == 0) { ++a; m /= 2; }
  while (m % 3 == 0) { ++b; m /= 3; }
  while (m % 5 == 0) { ++c; m /= 5; }
  Cover cover;
  cover.shapes = k == 0 ? kFxShapes : kRtShapes;
  cover.count = static_cast<int>(k == 0 ? sizeof(kFxShapes) / sizeof(GroupShape) : sizeof(kRtShapes) / sizeof(GroupShape));
  cover.cap = cap < 5 ? 5 : cap;
  for (int n = 0; n <= kFxPasses && cover.best_sum == INT_MAX; ++n) {
    if (n == 0 && a + b + c == 0) cover.best_sum = 0;
    else cover.search(a, b, c, 0, n, 0);
  }
  if (cover.best_sum == INT_MAX) return false;
  struct P {
    int id, ra, rb;
    int size() const { return ra * rb; }
  };
  std::vector<P> ps;
  for (int i : cover.best) {
    const GroupShape& g = cover.shapes[i];
    ps.push_back(P{g.id, g.r[0], g.r[1]});
  }
  std::stable_sort(ps.begin(), ps.end(), [](const P& x, const P& y) {
    if ((x.size() & 1) != (y.size() & 1)) return (x.size() & 1) > (y.size() & 1);
    return x.size() > y.size();
  });
  for (int p = 7; p <= kMaxGenericRadix && m > 1; p += 2)
    while (m % p == 0) {
      ps.push_back(P{FX_GENERIC, p, 1});
      m /= p;
    }
  if (m != 1 || static_cast<int>(ps.size()) > kFxPasses) return false;
  f.np = static_cast<int>(ps.size());
  // blocks after which a position is spared, and the positions of an index
  std::vector<int> spare;
  auto position = [&](int n) {
    int pos = n;
    for (int L : spare) pos += n / L;
    return pos;
  };
  int L = 1;
  for (const P& p : ps) {
    L *= p.size();
    if (L < M && L >= 8 && position(L) % 4 == 0) spare.push_back(L);
  }
  while (!spare.empty() && position(M - 1) + 1 > max_ls) spare.pop_back();
  f.ls = M > 0 ? position(M - 1) + 1 : 1;
  int lp = 1;
  std::vector<int> radix;
  for (int i = 0; i < kFxPasses; ++i) {
    FxPass& q = f.p[i];
    q = FxPass{};
    if (i >= f.np) {
      q.ulines = q.ulp = make_fastdiv(1);
      continue;
    }
    const int R = ps[i].size();
    q.shape = ps[i].id;
    q.R = R;
    q.lp = lp;
    q.step = position(lp);
    q.units = M / R;
    q.ts = M / (lp * R);
    q.ulines = make_fastdiv(static_cast<unsigned>(q.units));
    q.ulp = make_fastdiv(static_cast<unsigned>(lp));
    // Bits that the largest component may fill before the pass.  Magnitudes
    // then start below 2^(b + 1/2); a stage with twiddles multiplies them by
    // R / 4 at most, R of it before the factor 1/4 in a forward stage, and the
    // first pass's first stage has no factor.  A product's operand may reach
    // 2^62.8 (fx_cmul4's cross sums: 2^61.5 + 2^62.3 < 2^63), the results of the
    // last forward pass 2^62 (pairs of them are added).
    const bool gen = q.shape == FX_GENERIC, first = i == 0;
    auto bits = [](double limit, double growth) { return static_cast<int>(std::floor(limit - 0.5 - std::log2(growth))); };
    const double ra = ps[i].ra, rb = ps[i].rb;
    if (gen) {
      q.bits_dif = bits(first ? 62.0 : 62.8, R / 4.0);
      q.bits_dit = first ? bits(62.8, R / 4.0) : std::min(62, bits(62.8, std::max(1.0, R / 16.0)));
    } else {
      const double last = rb > 1 ? rb / 4 * ra : ra;   // forward: growth up to the sums of the last stage
      q.bits_dif = std::min(bits(62.8, rb > 1 ? rb : last), bits(first ? 62.0 : 62.8, last));
      q.bits_dit = first ? bits(62.8, ra) : 62;
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
      perm[n] = position(pos);
    }
  }
  if (nat_out) {
    nat_out->resize(M);
    for (int n = 0; n < M; ++n) (*nat_out)[n] = position(n);
  }
  return true;
}

int line_limit(int k, int M, int tile) {
  const int eb = k == 0 ? 16 : 8;
  const int T = tile > 1 ? tile : 1;
  // column_stride rounds a line up to `want` modulo `period`
  const int period = 128 / eb, want = T < period ? period / T : 1;
  const int most = static_cast<int>(kPassSmem / (static_cast<size_t>(T) * eb));
  int limit = most - ((most - want) & (period - 1));
  for (int lines = 1; lines <= 5; ++lines)
    if (row_admitted(M, lines, eb)) limit = std::min(limit, static_cast<int>(kPassSmem / (static_cast<size_t>(lines) * eb)));
  return limit;
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
  if (!group_plan(0, M, kGroupCap[0], p.fx, &t.perm_of[0], &t.nat_of[0], line_limit(0, M, 1)) ||
      !group_plan(1, M, kGroupCap[1], p.rt, &t.perm_of[1], &t.nat_of[1], line_limit(1, M, 1))) {
    set_error("internal: no passes for M=" + std::to_string(M));
    return GHB_ERR_INVALID;
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

ghb_status set_group_cap(PlanHolder& out, int k, int cap, int tile) {
  FftPlan& p = out.plan;
  FxPlan f = k == 0 ? p.fx : p.rt;
  std::vector<int> perm, nat;
  if (!group_plan(k, p.M, cap, f, &perm, &nat, line_limit(k, p.M, tile))) {
    set_error("internal: no passes for M=" + std::to_string(p.M));
    return GHB_ERR_INVALID;
  }
  perm.insert(perm.end(), nat.begin(), nat.end());
  GHB_CUDA_TRY(cudaMemcpy(out.d_group_perm[k], perm.data(), sizeof(int) * perm.size(), cudaMemcpyHostToDevice));
  GHB_CUDA_TRY(cudaStreamSynchronize(cudaStreamLegacy));   // in place before any stream's kernels read it
  (k == 0 ? p.fx : p.rt) = f;
  out.cap[k] = cap;
  return GHB_OK;
}

ghb_status make_plan_untuned(int M, PlanHolder& out) {
  PlanTables t;
  ghb_status st = build_plan_tables(M, out.plan, t);
  if (st != GHB_OK) return st;
  FftPlan& p = out.plan;
  // all tables in one block, copied at once (one allocation, copy and wait: an image
  // context makes plans at every change of its image)
  std::vector<char> h;
  auto put = [&h](const auto& v) {
    const size_t at = h.size();
    h.resize((at + sizeof(v[0]) * v.size() + 255) & ~static_cast<size_t>(255));
    std::memcpy(h.data() + at, v.data(), sizeof(v[0]) * v.size());
    return at;
  };
  size_t group[2];
  for (int k = 0; k < 2; ++k) {
    std::vector<int> both = t.perm_of[k];
    both.insert(both.end(), t.nat_of[k].begin(), t.nat_of[k].end());
    group[k] = put(both);
  }
  const size_t fx = put(t.fx_tw), tw = put(t.tw32);
  const bool ct = ct_size(M) && ct_plan(M).ok;
  std::vector<int> pct(ct ? M : 0);
  if (ct) ct_perm(M, pct.data());
  const size_t perm_ct = put(pct);
  GHB_CUDA_TRY(cudaMalloc(&out.d_tables, h.size()));
  GHB_CUDA_TRY(cudaMemcpy(out.d_tables, h.data(), h.size(), cudaMemcpyHostToDevice));
  GHB_CUDA_TRY(cudaStreamSynchronize(cudaStreamLegacy));   // a pageable copy: in place before other streams read
  for (int k = 0; k < 2; ++k) {
    out.d_group_perm[k] = reinterpret_cast<int*>(out.d_tables + group[k]);
    out.cap[k] = kGroupCap[k];
    FxPlan& f = k == 0 ? p.fx : p.rt;
    f.perm = out.d_group_perm[k];
    f.nat = out.d_group_perm[k] + M;
  }
  p.fx.tw = reinterpret_cast<const fxw*>(out.d_tables + fx);
  p.rt.tw32 = reinterpret_cast<const float2*>(out.d_tables + tw);
  p.ct = CtTables{ct ? reinterpret_cast<const int*>(out.d_tables + perm_ct) : nullptr, p.rt.tw32};
  p.ct_col = p.ct_row = p.ct_row3 = ct ? 1 : 0;
  return GHB_OK;
}

void free_plan(PlanHolder& p) {
  if (p.d_tables) cudaFree(p.d_tables);
  p = PlanHolder{};
}

}  // namespace ghb
