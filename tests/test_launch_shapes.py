"""What the pass launchers of csrc/passes.cu decide, on the host: the library's own
dispatch code with recorders in place of the kernels' launchers."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1412_2033_gb300", "csrc")

RECORDERS = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include "passes_fx.cuh"
#include "passes_rt.cuh"
namespace ghb {
std::string error_text;
int last_lines = 0, last_rows = 0, launched = 0;
size_t last_smem = 0;
void set_error(const std::string& s) { error_text = s; }
ghb_status apply_tune(int, PlanHolder&) { return GHB_OK; }
template <int M> ghb_status launch_col_ct_m(int, int, const ColArgs&, const CtTables&, cudaStream_t) { return GHB_OK; }
template <int M> ghb_status launch_row_ct_m(int, const RowArgs&, const CtTables&, int, cudaStream_t) { return GHB_OK; }
#define CT(m) template ghb_status launch_col_ct_m<m>(int, int, const ColArgs&, const CtTables&, cudaStream_t); \
  template ghb_status launch_row_ct_m<m>(int, const RowArgs&, const CtTables&, int, cudaStream_t);
CT(162) CT(486) CT(1458) CT(4374) CT(2187) CT(72) CT(135) CT(270)
ghb_status col(const FxPlan& f, int TW, int eb) {
  ++launched;
  last_lines = TW;
  last_smem = static_cast<size_t>(TW) * column_stride(f.ls, TW, eb) * eb;
  return GHB_OK;
}
ghb_status row(const FxPlan& f, int rows, int lines, int eb) {
  ++launched;
  last_rows = rows;
  last_lines = lines;
  last_smem = static_cast<size_t>(lines) * f.ls * eb;
  return GHB_OK;
}
ghb_status launch_fx_col(int, const ColArgs&, const FxPlan& f, int TW, cudaStream_t) { return col(f, TW, 16); }
ghb_status launch_rt_col(int, const ColArgs&, const FxPlan& f, int TW, cudaStream_t) { return col(f, TW, 8); }
ghb_status launch_fx_row(int, const RowArgs&, const FxPlan& f, int r, int n, int, cudaStream_t) { return row(f, r, n, 16); }
ghb_status launch_rt_row(const RowArgs&, const FxPlan& f, int r, int n, cudaStream_t) { return row(f, r, n, 8); }
ghb_status launch_fx_col_batch(int, const ColItem*, int, int64_t, size_t, int, cudaStream_t) { return GHB_OK; }
ghb_status launch_rt_col_batch(int, bool, const ColItem*, int, int64_t, size_t, int, cudaStream_t) { return GHB_OK; }
ghb_status launch_fx_row_batch(int, const RowItem*, int, int64_t, size_t, int, cudaStream_t) { return GHB_OK; }
ghb_status launch_rt_row_batch(const RowItem*, int, int64_t, size_t, int, cudaStream_t) { return GHB_OK; }
}  // namespace ghb
using namespace ghb;
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    """run(body, *arguments): the words that main() { body } prints."""
    tmp = tmp_path_factory.mktemp("launch_shapes")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    flags = [nvcc, "-O2", "-std=c++17", "-w", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
             os.path.join(ROOT, "include")]
    objects = []
    for unit in ("passes", "plan"):
        objects.append(str(tmp / f"{unit}.o"))
        subprocess.run([*flags, "-c", "-o", objects[-1], os.path.join(CSRC, unit + ".cu")], check=True)

    def go(body, *arguments):
        name = tmp / f"t{abs(hash(body))}"
        (tmp / (name.name + ".cu")).write_text(RECORDERS + "int main(int argc, char** argv) {" + body + "}")
        subprocess.run([*flags, "-o", str(name), str(name) + ".cu", *objects], check=True)
        return subprocess.run([str(name), *map(str, arguments)], capture_output=True, text=True, check=True).stdout.split()

    return go


def test_column_offsets_are_bounded_by_one_outer_index(run):
    """The FP32 column pass adds 32-bit row offsets to a 64-bit base: operands of 2^31
    entries and more run as long as the rows of one outer index stay below (d = 3
    axes at M = 1440 and 2560); beyond, the call is refused."""
    out = run(r"""
      auto ask = [](int64_t outer, int M, int N, int64_t inner) {
        FftPlan p{};
        group_plan(1, M, 32, p.rt, nullptr, nullptr);
        p.M = M;
        for (int sign : {+1, -1}) {
          ColArgs a{};
          a.outer = outer;
          a.inner = inner;
          a.Lin = sign > 0 ? N : M;
          a.Lout = sign > 0 ? M : N;
          launched = 0;
          const ghb_status st = launch_col<float>(sign, COL_PLAIN, a, p, nullptr);
          printf("%d%d ", st == GHB_OK, launched);
        }
      };
      ask(3 * 1440, 1440, 715, 358);                    // axis 2 at N = 715: 2.2e9 entries
      ask(3 * 2560LL, 2560, 1279, 640);                 // axis 2 at the largest order
      ask(3, 2560, 1279, 1279LL * 640);                 // axis 1 there: 2095513600 entries an outer index
      ask(1, 2048, 1023, (int64_t(1) << 31) / 2048 - 1);
      ask(1, 2048, 1023, (int64_t(1) << 31) / 2048);    // 2^31 entries: refused
    """)
    assert out == ["11"] * 8 + ["00"] * 2


def test_every_admitted_length_and_tile_fits_shared_memory(run):
    """Lengths with primes up to 31, every group size: what the size rules admit
    (columns of one line, forced tiles, rows) is launched as asked, in the kernels'
    220 KB, and with lines whose entries are evenly spaced in every group.  One length
    more than that is refused with a message."""
    out = run(r"""
      int bad = 0, dropped = 0, launches = 0;
      for (int M = 1; M <= 27000; ++M) {
        if (!factorizable(M)) continue;
        for (int k = 0; k < 2; ++k)
          for (int cap : {5, 8, 9, 10, 16, 32}) {
            const int eb = k == 0 ? 16 : 8;
            FftPlan p{};
            p.M = M;
            FxPlan& f = k == 0 ? p.fx : p.rt;
            std::vector<int> pos;
            for (int tile : {0, 1, 2, 4, 8, 16}) {
              if (tile == 0) group_plan(k, M, cap, f, nullptr, nullptr, line_limit(k, M, 1));
              if (tile > 0 && !col_admitted(M, tile, eb)) continue;
              if (f.ls > line_limit(k, M, tile)) {     // as tune.cu does for a forced tile
                ++dropped;
                group_plan(k, M, cap, f, nullptr, &pos, line_limit(k, M, tile));
                std::vector<char> seen(f.ls, 0);
                for (int n = 0; n < M; ++n) bad += pos[n] < 0 || pos[n] >= f.ls || seen[pos[n]]++;
                for (int i = 0; i < f.np; ++i)
                  for (int u = 0, q; u < f.p[i].units; ++u)
                    for (int j = 0, e = fx_unit_entry(f.p[i], u, q); j < f.p[i].R; ++j)
                      bad += pos[e] + j * f.p[i].step != pos[e + j * f.p[i].lp];
              }
              p.tile[k] = tile;
              for (int64_t columns : {1, 50000}) {
                ColArgs a{};
                a.outer = 1;
                a.inner = columns;
                a.Lin = M;
                a.Lout = M;
                launched = 0;
                const ghb_status st = k == 0 ? launch_col<double>(-1, COL_PLAIN, a, p, nullptr) : launch_col<float>(-1, COL_PLAIN, a, p, nullptr);
                launches += launched;
                if (!col_admitted(M, 1, eb)) bad += st == GHB_OK || launched || error_text.find("too large") == std::string::npos;
                else bad += st != GHB_OK || launched != 1 || last_smem > kPassSmem || (tile > 0 && last_lines != tile);
              }
            }
            group_plan(k, M, cap, f, nullptr, nullptr, line_limit(k, M, 1));
            for (int d : {2, 3})
              for (int mode : {ROW_MATVEC, ROW_TOREAL, ROW_ENERGY})
                for (int64_t rows : {1, 5, 100000}) {
                  if (k == 1 && mode != ROW_MATVEC) continue;
                  RowArgs a{};
                  a.nfields = mode == ROW_ENERGY ? d : 1;
                  a.ncomp = mode == ROW_TOREAL ? 1 : d;
                  a.rows = rows;
                  int r, n;
                  row_lines(mode, a.nfields, a.ncomp, M, 0, &r, &n);
                  launched = 0;
                  const ghb_status st = k == 0 ? launch_row<double>(mode, a, p, nullptr) : launch_row<float>(mode, a, p, nullptr);
                  launches += launched;
                  if (!row_admitted(M, n, eb)) bad += st == GHB_OK || launched || error_text.find("too large") == std::string::npos;
                  else bad += st != GHB_OK || launched != 1 || last_smem > kPassSmem;
                }
          }
      }
      printf("%d %d %d", bad, dropped > 100, launches > 100000);
    """)
    assert out == ["0", "1", "1"]


def test_forced_rows_are_launched(run):
    """rows32 of ghb_tune_set is what a d = 2 FP32 last-axis pass launches, at every
    length whose two lines are admitted."""
    out = run(r"""
      int bad = 0, n = 0;
      for (int M = 1; M <= 13000; ++M) {
        if (!factorizable(M) || !row_admitted(M, 2, 8)) continue;
        FftPlan p{};
        p.M = M;
        group_plan(1, M, 32, p.rt, nullptr, nullptr, line_limit(1, M, 1));
        for (int rows : {1, 2}) {
          p.rows32 = rows;
          RowArgs a{};
          a.nfields = 1;
          a.ncomp = 2;
          a.rows = 100;
          bad += launch_row<float>(ROW_MATVEC, a, p, nullptr) != GHB_OK || last_rows != rows || last_smem > kPassSmem;
          ++n;
        }
      }
      printf("%d %d", bad, n > 1000);
    """)
    assert out == ["0", "1"]


def test_last_axis_choices_of_two_and_three_components(run):
    """The autotuner times d = 2 and d = 3 last-axis passes apart: each takes the
    size-specialised kernels by its own flag."""
    out = run(r"""
      FftPlan p{};
      p.M = 162;
      group_plan(1, 162, 32, p.rt, nullptr, nullptr, line_limit(1, 162, 1));
      int some = 0;
      p.ct.perm = &some;
      for (int d : {2, 3})
        for (int two : {0, 1})
          for (int three : {0, 1}) {
            RowArgs a{};
            a.nfields = 1;
            a.ncomp = d;
            a.rows = 100000;
            a.H = 41;
            p.ct_row = two;
            p.ct_row3 = three;
            launched = 0;                       // run-time launches; the specialised ones are not counted
            launch_row<float>(ROW_MATVEC, a, p, nullptr);
            printf("%d", launched);
          }
    """)
    assert out == ["11001010"]
