"""The benchmark's result line is short enough to be read back from the tail of its output, whatever was measured beside it."""
import json

import bench


def _line(n):
    roof = {"kernel": "k" * 40, "bound": "tensor", "achieved": 1.0, "peak": 2.0, "unit": "TFLOP/s", "frac": 0.5, "note": "n" * 200}
    return {"metric": bench.METRIC, "value": 812.3, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": 19.7,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
            "config": {"workload": bench.WORKLOADS["cfg5"], "cache": "c" * 200, "parallelism": "p" * 40},
            "repeats": {"n": 5, "ms_per_step": [19.7] * 5}, "clocks": {"sm_mhz": 1965, "sm_max_mhz": 1965, "reasons": []},
            "e2e": {"value": 800.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 4}, "gpu_launches": 5000,
            "roofline": roof, "rooflines": {str(i): roof for i in range(n)}, "roofline_update": roof, "gemm_all": roof, "elementwise": roof,
            "kernel_ms_per_step": {str(i): 1.0 for i in range(n)},
            "other_workloads": [{"workload": w, "value": 1.0, "rooflines": {str(i): roof for i in range(n)}} for w in bench.WORKLOADS.values()],
            "variants": [{"option": "materialize_backward", "value": 830.0, "rooflines": {}}, {"option": "x", "error": "no memory"}],
            "cpu_baseline": {"value": 0.07, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 300},
            "update_sweep": [{"n_params": 10 ** 6, "P": p, "ms": 0.01} for p in range(n)]}


def test_split():
    for n in (1, 40):
        line = _line(n)
        brief, detail = bench.split_line(line)
        assert len(json.dumps(brief)) <= bench.LINE_BYTES
        for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                    "data", "config", "clocks", "e2e", "gpu_launches"):
            assert brief[key] == line[key]
        assert brief["variants"] == {"materialize_backward": 830.0, "x": "error"}
        assert set(line) == set(brief) | set(detail)
        for key in ("rooflines", "update_sweep", "other_workloads"):
            assert detail[key] == line[key]
