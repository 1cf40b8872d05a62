"""bench.py's line: the contract's keys, short enough for readers that keep a few
KB of output, without the details that go to stderr."""
import json

import bench


def test_short_line():
    kern = {f"kernel_{k}": {"achieved": 1.25, "peak": 77.1, "unit": "TFLOP/s", "ms": 3.5} for k in range(40)}
    form = {"value": 1.0e9, "ms_per_step": 5.0, "steps": 3, "kernels": kern}
    config = {"value": 2.0e9, "ms_per_step": 1.5, "chosen_form": "mixed_full", "kernels": kern,
              "fp64_form": form, "forms": {"mixed": form}, "accuracy": {"bound": 1e-6, "max_err": 3e-7}}
    line = {"metric": "m", "value": 9.0e9, "unit": "entries/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 59.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic", "config": {"workload": "w"}, "roofline": {"frac": 0.6},
            "e2e": {"value": 2.0e9, "unit": "entries/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
            "gpu_launches": 320, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "kernels": kern, "fp64_form": form, "forms": {"mixed": form}, "work": {"pairs": 1},
            "configs": {f"C{k}": config for k in range(5)}, "green_matrices": {"laplace_slp": form}}
    got = bench.short_line(line)
    for k, v in line.items():
        if k not in ("kernels", "forms", "work", "fp64_form", "configs", "green_matrices"):
            assert got[k] == v
    assert got["fp64_form"] == {"value": 1.0e9, "ms_per_step": 5.0, "steps": 3}
    assert got["configs"]["C0"]["value"] == 2.0e9
    assert got["configs"]["C0"]["accuracy"] == {"bound": 1e-6, "max_err": 3e-7}
    assert "kernel_0" not in json.dumps(got)
    assert len(json.dumps(got)) < 4000
    assert "kernel_0" in json.dumps(line)      # the details stay whole
