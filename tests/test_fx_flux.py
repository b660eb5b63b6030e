"""The FP64 mode's fixed-point two-point flux (csrc/es_fx.cuh) against the same formulas in long
double on the host, over gas constants, Mach numbers, jumps up to the branch limits and values next
to powers of two; and the states that must leave the fixed-point path.

Bound: a component is a sum of at most two products whose factors each carry a few units of their
last bit, amplified by at most 1/S1 < 3 and the four-fold shifts: 64 units of the result's last
bit (2^-61 or 2^-62 of the block scale), beside the 2^-53 of the value.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("fx") / "check")
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-O2", "-I",
                    os.path.join(ROOT, "paper_2003_08831_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx_flux_check.cu")], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()


def test_flux_against_long_double(lines):
    pairs = [ln.split() for ln in lines if ln.startswith("pair")]
    assert len(pairs) == 4 * 7 * 5
    for ln in pairs:
        assert int(ln[5]) == 0, ln  # all in range: the fixed-point path is taken
        assert max(map(float, ln[7:10])) <= 64.0, ln


def test_states_outside_the_range(lines):
    bad = [ln for ln in lines if ln.startswith("bad")]
    assert bad == ["bad 0"] * 12
