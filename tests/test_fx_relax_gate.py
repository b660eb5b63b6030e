"""The relaxation's early decisions (csrc/es_relax_fx.cuh) against long double on the host: no element whose
RMS change is above the floor is taken for unconstrained by its largest increment, and a quadratic root
inside the solver's range 0.5 .. 1.5 is never refused (outside 0.498 .. 1.502 always: the estimates carry
20 bits, 2^-19 in all)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


def test_floor_and_root_range(tmp_path):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "check")
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-O2", "-I",
                    os.path.join(ROOT, "paper_2003_08831_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx_relax_gate_check.cu")], check=True)
    rows = [ln.split() for ln in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    floor, near = [r for r in rows if r[0] == "floor"], [r for r in rows if r[0] == "near"]
    assert len(floor) == len(near) == 4
    for r in floor:
        assert int(r[3]) > 1000 and int(r[5]) == 0 and r[7] == "1", r
    for r in near:
        assert int(r[3]) > 1000 and int(r[5]) == 0 and int(r[7]) == 0, r
