"""A thread's part of an inner product (ThreadSum, csrc/reduce.cuh) on the host."""
import os
import shutil
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "reduce.cuh"
int main() {
  std::mt19937 rng(7);
  std::uniform_real_distribution<float> u(0.0f, 1.0f);
  for (int n : {1, 2, 8, 16, 1000, 100000}) {
    double worst = 0;
    for (int repeat = 0; repeat < 20; ++repeat) {
      ghb::ThreadSum<float, true> sum;
      double exact = 0;
      for (int i = 0; i < n; ++i) {
        const float s = std::ldexp(u(rng), int(rng() % 12));   // entries of an inner product, of mixed size
        sum.close(sum.open() + s);
        exact += s;
      }
      worst = std::fmax(worst, std::fabs(sum.total() - exact) / exact);
    }
    printf("%d %.3e\n", n, worst);
  }
}
"""


def test_entries_are_added_without_fp32_rounding(tmp_path):
    """Two-sum leaves an error of the second float only: at most n 2^-24 of n 2^-24 of
    the sum of positive entries, and two roundings to double in this check; a plain
    FP32 sum of eight entries is off by 2^-24 and more."""
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "sum.cu", tmp_path / "sum"
    src.write_text(SOURCE)
    subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I",
                    os.path.join(ROOT, "paper_1412_2033_gb300", "csrc"), "-o", str(exe), str(src)], check=True)
    rows = [r.split() for r in subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    assert len(rows) == 6
    for n, error in rows:
        n = int(n)
        assert float(error) <= (n * 2.0 ** -24) ** 2 + n * 2.0 ** -53, (n, error)
