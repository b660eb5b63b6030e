"""The entropy-variable increment w(u + e) - w(u) of the FP64 and ES_MIXED modes in fixed point
(csrc/es_prep_fx.cuh) against long double on the host, for changes of 1e-13 to 2e-2 of the state.

Bounds.  A component is a sum of products of at most six factors and partial sums, each good to 2^-58
of itself or of the largest term of its sum: 6 2^-58 = 0.19 units of 2^-53 of the terms' sizes, below 0.25,
beside the result's own rounding.  Relative to the component itself the mean error is no larger than
that of the same formula in double.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def test_increment_against_long_double(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "check")
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-O2", "-I",
                    os.path.join(ROOT, "paper_2003_08831_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx_increment_check.cu")], check=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()
    rows = [ln.split() for ln in lines if ln.startswith("increment")]
    assert len(rows) == 5 * 6 * 6
    for ln in rows:
        # (rho p changes by up to two times the state's change; some of the largest leave the range)
        assert int(ln[5]) == 0 or float(ln[3]) > 8e-3, ln
        assert int(ln[5]) <= 2000, ln
        assert float(ln[7]) <= 0.25, ln
        means = list(map(float, ln[9:19]))
        for fixed, double in zip(means[::2], means[1::2]):
            assert fixed <= double, ln
    assert [ln for ln in lines if ln.startswith("bad")] == ["bad 0"] * 12
    assert "wide 0" in lines  # changes of rho or rho p beyond 2 %, up to a factor 5
    zero = [ln.split() for ln in lines if ln.startswith("zero")]
    assert len(zero) == 1 and zero[0][1] == "1" and all(float(v) == 0.0 for v in zero[0][2:])
