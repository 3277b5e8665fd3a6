"""bench.py's result line keeps the fields its readers need and stays short."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def _full():
    """What run_ours measures, with long prose wherever it has prose."""
    prose = "x" * 400
    leg = {"products_per_s": 123456789.123, "path": prose, "bit_exact_sample": True}
    return {
        "metric": bench.METRIC, "value": 246556879.74008718, "unit": "products/s", "n_gpus": 1, "steps": 20, "warmup": 5,
        "ms_per_step": 0.016612799465656282, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "u32", "data": "synthetic (seeded uniform residues)",
        "config": {"workload": bench.WORKLOAD, "path": "ntt", "autotuned": {"note": prose}, "overlap": "y" * 80,
                   "n": 1024, "q": [12289], "batch": 4096, "l2": "z" * 80, "parallelism": "single"},
        "e2e": {"value": 2.2e7, "unit": "products/s", "h2d_bytes_per_step": 33554432, "d2h_bytes_per_step": 16777216,
                "api": "polymul_batch_mapped on page-locked host buffers: " + prose, "roofline": None,
                "per_call_sync": {"value": 1.0 / 3}, "staged": {"value": 2.0 / 3}, "host_link": {"note": prose}},
        "gpu_launches": 20,
        "roofline": {"bound": "alu", "achieved": 4039.58, "peak": 5034.24, "unit": "Gmulmod/s", "frac": 0.8,
                     "traffic": None, "kernel": "k_ntt_batch<u32> (" + prose, "work": prose, "hbm": {"frac": 0.45}},
        "cpu_baseline": {"value": 1.4e4, "unit": "products/s", "cores": 16, "kind": "oracle", "sample": prose},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 5},
        "bit_exact_sample": True,
        "tensor_path": {"value": 5e7, "unit": "products/s", "roofline": {"frac": 0.21}, "bit_exact_sample": True},
        "other_workloads": dict({"leg_%d" % i: leg for i in range(9)},
                                crossover={"rows": [prose] * 9, "bit_exact_sample": True},
                                serve_20k={"requests": 20000, "saturated": {"seconds": 0.73}, "bit_exact_sample": True}),
    }


def test_line_is_short_and_complete():
    line = bench.summary_line(_full())
    text = json.dumps(line)
    assert len(text) < 3000 and "\n" not in text
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks", "roofline", "cpu_baseline"):
        assert key in line, key
    assert line["value"] == 246556879.74008718
    assert line["e2e"]["h2d_bytes_per_step"] == 33554432 and line["e2e"]["d2h_bytes_per_step"] == 16777216
    assert line["clocks"]["sm_mhz"] == 2070.0


def test_line_without_the_optional_legs():
    full = _full()
    full.update(tensor_path=None, other_workloads=None, cpu_baseline=None)
    line = bench.summary_line(full)
    assert line["tensor_path"] is None and line["other_workloads"] is None and line["cpu_baseline"] is None
