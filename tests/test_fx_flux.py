"""The FP64 mode's fixed-point two-point flux (csrc/es_fx.cuh), interface flux, parameter vector
and entropy-variable increment (csrc/es_*_fx.cuh) against the same formulas in long
double on the host, over gas constants, Mach numbers, jumps up to the branch limits and values next
to powers of two; and the states that must leave the fixed-point path.

Bound: a component is a sum of at most two products whose factors each carry a few units of their
last bit, amplified by at most 1/S1 < 3 and the four-fold shifts: 64 units of the result's last
bit (2^-61 or 2^-62 of the block scale), beside the 2^-53 of the value.  The parameter vector: 2^-53
from the rounding to a double, and 2^-58 beside it (times the ratio of rho E to the internal
energy, below 7 here).  The increment is a difference of values good to 2^-58 of their scale, at
most eight of which enter: 2^-55, a quarter of 2^-53, beside the double's half unit of a change
below 0.02.  The interface flux (csrc/es_face_fx.cuh): flux, dissipation and their difference are
rounded to doubles once each, 2^-53 of their scale, and the flux itself is good to 2^-53 of its own
as above: four of them.
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
    outq = [ln for ln in lines if ln.startswith("outq")]
    assert outq == ["outq 0"] * 10


def test_parameter_vector_and_increment(lines):
    rows = [ln.split() for ln in lines if ln.startswith("state")]
    assert len(rows) == 3 * 4 * 3
    for ln in rows:
        # outside the range: the fastest flows (it ends by exponents, between |z_v| = 1 and 4), and some
        # of the quarter of the states that are placed at powers of two, where the scales change
        assert int(ln[5]) <= 100, ln
        assert float(ln[7]) <= 1.0 + 7.0 / 32.0, ln
        assert float(ln[8]) <= 0.25 + 0.02, ln


def test_interface_flux(lines):
    rows = [ln.split() for ln in lines if ln.startswith("face")]
    assert len(rows) == 3 * 2 * 4 * 4
    for ln in rows:
        assert int(ln[6]) == 0 or float(ln[4]) == 2.5, ln
        assert float(ln[8]) <= 4.0, ln
