"""The fixed-point two-point flux (csrc/es_fx.cuh) at the edges of its range, on the host against long double.

Bounds.
* Slow gas: the factors of mass and energy flux carry units of 2^-62 of the block scale, 64 of them in all
  (tests/test_fx_flux.py); with |Q_ij| >= 1/4, velocity and z5 at least half of their blocks' the mass flux is above
  2^-4 of the scale and the energy flux above 2^-6, so 64 units are 2 and 8 units of 2^-53 of the flux itself.
* Room beyond an element's scales: no more than three bits above what its fluxes need, of the five that the sums
  have over a double's.
* Near tier: the correction is good to five units of 2^-53 at its limit (the sum of its roundings stands beside it
  in the header), and the flux is no further from long double than the FP64 kernels' form of it, on average and
  at worst.
* Metrics: where they are taken, the sums are no further off than the same sums in FP64.
* Line sums: below 2^63 for the operators' own Q_ij with the largest face flux that is taken.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"


@pytest.fixture(scope="module")
def check(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    exe = str(tmp_path_factory.mktemp("fx") / "check")
    subprocess.run([NVCC, "-std=c++17", "--expt-relaxed-constexpr", "-w", "-O2", "-I",
                    os.path.join(ROOT, "paper_2003_08831_gb300", "csrc"), "-o", exe,
                    os.path.join(ROOT, "tests", "fx_pair_check.cu")], check=True)

    def run(part):
        out = subprocess.run([exe, part], check=True, capture_output=True, text=True).stdout
        return [ln.split() for ln in out.splitlines()]
    return run


def test_slow_gas(check):
    rows = check("slow")
    assert len(rows) == 4 * 6 * 3
    for ln in rows:
        assert int(ln[5]) == 0, ln
        assert float(ln[7]) <= 2.0 and float(ln[9]) <= 8.0, ln


def test_room_for_larger_fluxes(check):
    # what the fluxes need and three bits beside it, up to 2^6 times the pressure and the enthalpy flux at sound speed
    (row,) = check("room")
    assert int(row[2]) == 0 and int(row[4]) > 1000 and int(row[6]) > 1000, row


def test_near_tier_to_its_limit(check):
    rows = check("near")
    assert rows[0][0] == "correction" and int(rows[0][1]) > 100000
    assert float(rows[0][3]) <= 5.0, rows[0]
    assert len(rows) == 1 + 4 * 4
    for ln in rows[1:]:
        assert int(ln[4]) > 10000, ln
        values = list(map(float, ln[5:13]))  # mean mass, energy; largest mass, energy: fixed point, FP64
        for fixed, double in zip(values[::2], values[1::2]):
            assert fixed <= double, ln


def test_line_sums(check):
    rows = check("sums")
    assert len(rows) == 4
    for ln in rows:
        assert int(ln[3]) == 0 and int(ln[5]) > 0, ln
        assert int(ln[7]) == 0, ln          # every sum beyond 2^61 is seen
        assert float(ln[9]) < 1.0, ln       # none passes 2^63
        assert float(ln[11]) < 0.98, ln


def test_metrics(check):
    rows = check("metrics")
    assert len(rows) == 4 * 8
    for ln in rows:
        taken, ratio = int(ln[4]), float(ln[2])
        assert taken == (ratio < 17.0), ln  # 1.9 and 1.9 ratio: exponents up to four apart
        if taken:
            for fixed, double in zip(ln[5::2], ln[6::2]):
                assert float(fixed) <= float(double), ln
