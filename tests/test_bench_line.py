"""The benchmark's printed line: every key of its contract, and short enough (below 3000 characters with every
form) to be kept whole by a log that holds the end of the output; the rooflines
of modes whose FP64 work runs on the integer pipe are of HBM or the FP32 pipe."""
import json
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
KEYS = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
        "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks", "e2e")


def test_printed_line():
    sys.path.insert(0, ROOT)
    import bench
    rate = 4131321231.2134567
    form = {"value": rate, "ms_per_step": 1.523423423, "speedup_vs_fp64_same_physics": 2.17412341,
            "kernel_roofline": {"volume": {"bound": "hbm", "frac": 0.41212341}},
            "error_vs_fp64": {"rel_l2": 9.5755395e-08},
            "degree_mix": {"predicted_from_degree_mix": rate, "measured_over_predicted": 0.9971234}}
    out = {"metric": bench.METRIC, "value": rate, "unit": bench.UNIT, "n_gpus": 8, "steps": 2000, "warmup": 50,
           "ms_per_step": 1.523423423, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic (closed-form Taylor-Green vortex, Mach 0.1)", "config": bench.workload_config(bench.MAIN),
           "gpu_launches": 27200, "kernel_share": {"volume": 0.5}, "forms": {"x": form}, "dt": 0.1,
           "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"], "samples": 1500},
           "e2e": {"value": rate, "unit": bench.UNIT, "h2d_bytes_per_step": 83886088, "d2h_bytes_per_step": 83886096,
                   "ms_per_step": 2.3123123},
           "kernel_roofline": {"volume": {"bound": "hbm", "frac": 0.23121, "frac_hbm": 0.23121}},
           "cpu_baseline": {"value": rate, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "x" * 300},
           "short": {k: bench.compact(form) for k in ("ns_fp64", "ns_mixed", "ns_mixed_ff", "ns_fp64x", "euler_mixed",
                                                      "euler_mixed_ff", "euler_fp64x", "batch_fp64", "batch_mixed_ff")}}
    text = json.dumps(bench.printed(out))
    assert len(text) < 3000
    line = json.loads(text)
    assert all(k in line for k in KEYS) and line["value"] == rate and "kernel_share" not in line
    assert len(line["forms"]) == 9 and line["forms"]["ns_fp64"]["value"] == pytest.approx(rate, rel=1e-3)


def test_fixed_point_rooflines():
    sys.path.insert(0, ROOT)
    import bench
    peaks = {"fp64_tflops": 1.0, "fp32_tflops": 64.0}
    kr = bench.kernel_rooflines(3, 1000, 0, {k: (1.0, 10) for k in ("prep", "face", "volume", "relax")}, peaks)
    for k, v in bench.fixed_point_rooflines(kr).items():
        assert v["bound"] in ("hbm", "fp32") and v["fp64_equivalent"] == kr[k]["frac_fp64"]
        assert v["frac"] == max(kr[k]["frac_hbm"], kr[k]["frac_fp32"]) and "frac_fp64" not in v
