"""The fixed-point transform on the host (as in test_fx_emulation.py) with the lines
that grow most: full-magnitude constants, alternating signs and single frequencies."""
import os
import shutil
import subprocess

import pytest

from test_fx_emulation import CSRC, ROOT, SOURCE

DATA = "x[k] = kind == 0 ? z : kind == 1 ? z / (1.0 + std::abs(f)) : z * 1e-3 + (k == 0 ? 1.0 : 0.0);"
EXTREME = """
          const double most = 1.0 - 0x1p-53;               // full magnitude in both components
          const double t = 2 * M_PI * ((long long)k * (M / 3 + 1) % M) / M;
          x[k] = kind == 0 ? Z<double>(most, most) : kind == 1 ? (k % 2 ? -1.0 : 1.0) * Z<double>(most, -most)
                                                                 : Z<double>(std::cos(t) > 0 ? most : -most, std::sin(t) > 0 ? most : -most);"""


@pytest.mark.parametrize("cap", [5, 9, 18])
def test_lines_of_full_magnitude_stay_in_range(tmp_path, cap):
    assert SOURCE.count(DATA) == 1
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    src, exe = tmp_path / "range.cu", tmp_path / "range"
    src.write_text(SOURCE.replace(DATA, EXTREME))
    subprocess.run([nvcc, "-O2", "-std=c++17", "-w", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-o", str(exe), str(src), os.path.join(CSRC, "plan.cu")], check=True)
    lengths = [2, 3, 4, 5, 6, 7, 8, 10, 12, 13, 16, 25, 27, 31, 45, 49, 64, 81, 90, 121, 125, 198, 243, 256, 310, 625, 640,
               961, 1024, 1458, 2048, 2401, 3125, 4374, 6400]
    out = subprocess.run([str(exe), str(cap), *map(str, lengths)], capture_output=True, text=True, check=True).stdout
    rows = [line.split() for line in out.splitlines()]
    assert len(rows) == 6 * len(lengths)
    for M, kind, dit, out_of_range, fixed, double in rows:
        assert out_of_range == "0", (M, kind, dit)
        # four roundings of 2^-60 of the largest entry a pass, here the line's root mean
        # square and 2^-1/2 of its modulus, and the outputs' rounding to double
        assert float(fixed) <= 2.0 ** -53 + 2.0 ** -58 * 4 * int(M) ** 0.5, (M, kind, dit, fixed, double)
