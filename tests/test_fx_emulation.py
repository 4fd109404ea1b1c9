"""The fixed-point transform of csrc/fft_fx.cuh run on the host (its arithmetic
compiles for both sides) against an extended-precision DFT and the same DFT in
double: every pass grouping, both directions, and no value out of range."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1412_2033_gb300", "csrc")

SOURCE = r"""
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include "fft_fx.cuh"
#include "ghb_internal.cuh"
namespace ghb { void set_error(const std::string&) {} ghb_status apply_tune(int, PlanHolder&) { return GHB_OK; } }
using namespace ghb;
template <typename T> using Z = std::complex<T>;
template <typename T> void dft(std::vector<Z<T>>& x, int sign, const std::vector<UnitRoot>& R, int stride) {
  const int n = x.size(), M = R.size();
  if (n == 1) return;
  int p = 2;
  while (n % p) ++p;
  const int m = n / p;
  std::vector<std::vector<Z<T>>> sub(p, std::vector<Z<T>>(m));
  for (int i = 0; i < n; ++i) sub[i % p][i / p] = x[i];
  for (auto& s : sub) dft(s, sign, R, stride * p);
  for (int k = 0; k < n; ++k) {
    Z<T> a(0, 0);
    for (int q = 0; q < p; ++q) {
      const long long e = (long long)q * k % n * stride % M;
      a += sub[q][k % m] * Z<T>((T)R[e].c, (T)(sign * R[e].s));
    }
    x[k] = a;
  }
}
int main(int argc, char** argv) {
  std::mt19937_64 rng(5);
  std::normal_distribution<double> nd;
  for (int arg = 2; arg < argc; ++arg) {
    const int cap = atoi(argv[1]), M = atoi(argv[arg]);
    FxPlan P{};
    std::vector<int> perm, pos;
    std::vector<UnitRoot> R;
    std::vector<fxw> tw;
    if (!group_plan(0, M, cap, P, &perm, &pos)) return 1;
    unit_roots(M, R);
    fx_twiddles(R, tw);
    // positions: distinct, inside the line, evenly spaced in every group; the first
    // pass's unit r holds the natural indices r + (M / R) rev(j)
    std::vector<char> seen(P.ls, 0);
    bool laid = true;
    for (int n = 0; n < M; ++n) laid &= pos[n] >= 0 && pos[n] < P.ls && !seen[pos[n]]++;
    for (int i = 0; i < P.np; ++i)
      for (int u = 0; u < P.p[i].units; ++u)
        for (int j = 0, p; j < P.p[i].R; ++j)
          laid &= pos[fx_unit_entry(P.p[i], u, p)] + j * P.p[i].step == pos[fx_unit_entry(P.p[i], u, p) + j * P.p[i].lp];
    const int rb[] = {1, 1, 1, 1, 2, 2, 3, 2, 1};
    for (int r = 0; P.np && r < P.p[0].units; ++r)
      for (int j = 0, B = rb[P.p[0].shape], A = P.p[0].R / B; j < P.p[0].R; ++j)
        laid &= perm[r] + j == perm[r + P.p[0].units * (j % A * B + j / A)];
    if (!laid) return 2;
    for (int kind = 0; kind < 3; ++kind)        // white, 1/(1+|k|), one coefficient over 1e-3 noise
      for (int dit = 1; dit >= 0; --dit) {
        std::vector<Z<double>> x(M);
        std::vector<Z<long double>> ref(M);
        int E = 1, mag = 0, range = 0;
        for (int k = 0; k < M; ++k) {
          const int f = k <= M / 2 ? k : k - M;
          const Z<double> z(nd(rng), nd(rng));
          x[k] = kind == 0 ? z : kind == 1 ? z / (1.0 + std::abs(f)) : z * 1e-3 + (k == 0 ? 1.0 : 0.0);
          ref[k] = Z<long double>(x[k].real(), x[k].imag());
          E = std::max(E, std::max(fx_absword(x[k].real()), fx_absword(x[k].imag())) >> 20);
        }
        const int b = dit ? P.p[0].bits_dit : P.p[P.np - 1].bits_dif;
        std::vector<fx2> buf(P.ls, fx2{0, 0});
        auto nat = [&](int k) { return pos[k]; };
        for (int k = 0; k < M; ++k)
          buf[dit ? perm[k] : nat(k)] = fx2{fx_from_double(x[k].real(), E, b), fx_from_double(x[k].imag(), E, b)};
        int e = E - 1022 - b;
        for (int q = 0; q < P.np; ++q) {
          const int i = dit ? q : P.np - 1 - q;
          const FxPass& S = P.p[i];
          const int g = q == 0 ? 0 : (dit ? S.bits_dit : S.bits_dif) - fx_bitlen(mag);
          mag = 0;
          for (int u = 0; u < S.units; ++u) {
            int p;
            fx2* base = &buf[pos[fx_unit_entry(S, u, p)]];
            const int m = dit ? (i ? fx_run_unit<1, true, false>(S, base, g, p, M, tw.data()) : fx_run_unit<1, true, true>(S, base, g, p, M, tw.data()))
                              : (i ? fx_run_unit<-1, false, false>(S, base, g, p, M, tw.data()) : fx_run_unit<-1, false, true>(S, base, g, p, M, tw.data()));
            mag = std::max(mag, m);
          }
          e += 2 * fx_quarters(S.shape, i == 0) - g;
          range |= mag >= (q + 1 < P.np || dit ? 0x70000000 : 1 << 30);   // 2^62.8, 2^62 after the last forward pass
        }
        std::vector<Z<double>> dbl(x);
        dft(ref, dit ? 1 : -1, R, 1);
        dft(dbl, dit ? 1 : -1, R, 1);
        long double n = 0, ef = 0, ed = 0;
        const FxScale s = fx_scale_of(e);
        for (int k = 0; k < M; ++k) {
          const fx2 v = buf[dit ? nat(k) : perm[k]];
          n += std::norm(ref[k]);
          ef += std::norm(Z<long double>(fx_to_double(v.x, s), fx_to_double(v.y, s)) - ref[k]);
          ed += std::norm(Z<long double>(dbl[k].real(), dbl[k].imag()) - ref[k]);
        }
        printf("%d %d %d %d %.3Le %.3Le\n", M, kind, dit, range, sqrtl(ef / n), sqrtl(ed / n));
      }
  }
}
"""


@pytest.mark.parametrize("cap", [5, 9, 18])
def test_transform_error_against_extended_precision(tmp_path, cap):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src = tmp_path / "emulation.cu"
    src.write_text(SOURCE)
    exe = tmp_path / "emulation"
    subprocess.run([nvcc, "-O2", "-std=c++17", "-w", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-o", str(exe), str(src), os.path.join(CSRC, "plan.cu")], check=True)
    lengths = [2, 3, 4, 5, 6, 7, 8, 10, 16, 29, 31, 45, 62, 64, 90, 125, 135, 162, 198, 270, 374, 486, 512, 527, 625,
               640, 961, 1000, 1024, 1458, 2048, 2187, 3125, 4096, 4374, 6250, 6400]
    out = subprocess.run([str(exe), str(cap), *map(str, lengths)], capture_output=True, text=True, check=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 6 * len(lengths)
    for M, kind, dit, out_of_range, fixed, double in rows:
        assert out_of_range == "0", (M, kind, dit)
        # white and decaying data: no further off than the transform in double (a few
        # units of 2^-53 for either); one dominant coefficient: its ratio to the root
        # mean square, sqrt(M) at most, uses up the extra bits (four roundings of 2^-60
        # of it per pass).  Either way the outputs themselves are rounded to double.
        own = 2.0 ** -53
        limit = max(float(double), 2.5e-16) if kind != "2" else own + max(float(double), 2.0 ** -58 * 4 * int(M) ** 0.5)
        assert float(fixed) <= limit, (M, kind, dit, fixed, double)
