"""The viscous flux in fixed point (csrc/es_viscous_fx.cuh) of nodes whose gradients are far below what the
element's scales hold (interior nodes, smooth flow), against long double on the host.

Bound: that of tests/test_fx_viscous.py, 5 and 15 units of 2^-53 of the flux of a gradient of 2^62, where the
node's largest gradient is brought to between 2^61 and 2^62: twice as many of its own flux.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def test_small_gradients_against_long_double(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "check")
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-O2", "-I",
                    os.path.join(ROOT, "paper_2003_08831_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx_viscous_small_check.cu")], check=True)
    rows = [ln.split() for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 4 * 4
    for ln in rows:
        assert float(ln[4]) <= 10.0, ln
        assert float(ln[5]) <= 30.0, ln
