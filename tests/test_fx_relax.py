"""The fixed-point relaxation root (csrc/es_relax_fx.cuh) against long double on the host, over gas
constants, Mach numbers, sizes of the increment up to the branch limit, degrees and kinds of
increments (independent, acoustic, shear, one node twenty times the others); and the states and
increments that must leave the fixed-point path.

Bound: with 53-bit node quantities the FP64 form is off by up to a few units of 2^-53 for every one
of a node's dozen roundings that do not average out.  Here X, Y, W carry 58 bits, of which a Mach
number M costs the internal energy log2(1 + gam (gam-1) M^2/2) (below 3 for M <= 4 but for sums of three
components: 5), and Y is a difference of terms up to 2^(1 + M) larger than itself: 2^-58 times 2^5
times 8 in the worst case, 8 units of 2^-53, beside the 2^-53 of the result; the mean over elements
stays below 2 of them.
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
                    os.path.join(ROOT, "tests", "fx_relax_check.cu")], check=True)
    return subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()


def test_root_against_long_double(lines):
    rows = [ln.split() for ln in lines if ln.startswith("root")]
    assert len(rows) == 3 * 4 * 6 * 3
    for ln in rows:
        assert int(ln[6]) == 0, ln  # all in range: the fixed-point path is taken
        assert float(ln[8]) <= 16.0, ln
        assert float(ln[10]) <= 2.0, ln


def test_outside_the_range(lines):
    assert [ln for ln in lines if ln.startswith("outd")] == ["outd 0"] * 5
    assert [ln for ln in lines if ln.startswith("outu")] == ["outu 0"] * 8
