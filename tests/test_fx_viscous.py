"""The viscous flux in fixed point (csrc/es_viscous_fx.cuh) against long double on the host, for gradients
up to the largest the block scales hold, Mach numbers and positions of the node's z1 in the
element's range.

Bound, in units of 2^-53 of the flux that the largest gradients give, beside the result's rounding:
the stresses' sums carry 2^-56 (six bits of room) times the at most eight that z1 below the
element's largest costs a = 1/z1^2's companion v theta, and five terms of them: 5 units; the energy adds
three products of them with a velocity: 15.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def test_viscous_flux_against_long_double(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "check")
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-O2", "-I",
                    os.path.join(ROOT, "paper_2003_08831_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx_viscous_check.cu")], check=True)
    rows = [ln.split() for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 4 * 3
    for ln in rows:
        assert float(ln[4]) <= 5.0, ln
        assert float(ln[5]) <= 15.0, ln
