"""The float kernels' arguments hold no fixed-point tables: every launch copies its arguments, and a step of
the mixed float-float mode is 13 launches of 10 to 160 us."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
SOURCE = """#include <cstdio>
#include "es_device.cuh"
int main() {
  printf("%zu %zu\\n", sizeof(es::Params), sizeof(es::FxParams));
}
"""


def test_tables_are_apart(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "size.cu", str(tmp_path / "size")
    src.write_text(SOURCE)
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-I",
                    os.path.join(ROOT, "paper_2003_08831_gb300", "csrc"), "-o", exe, str(src)], check=True)
    plain, fixed = map(int, subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split())
    assert fixed - plain >= 8 * (36 + 6)  # Q_ij and 1/omega_i
    # two FP64 and four FP32 tables of 36, the weights, constants, one instance's geometry and pointers
    assert plain <= 2 * 36 * 8 + 4 * 36 * 4 + 6 * 8 + 12 * 4 + 6 * 8 + 6 * (8 + 4 + 8) + 5 * 4 + 64 + 64
