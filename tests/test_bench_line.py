"""The benchmark's line on stdout: what its readers look for, short enough to survive where only the end of the output is kept."""
import json

import bench


def test_contract_line_is_short_and_complete():
    x = 1234.56789012345
    kernel_ms = {k: x for k in ("attn_bwd", "dWqkv+dXn", "dWo+dA", "proj_qkv", "attn_fwd", "proj_o", "db+norm_bwd", "norm_fwd", "db", "rope_bwd")}
    one = {"ms_per_step": x, "tflops": x}
    full = {
        "metric": "fwd+bwd layer TFLOP/s", "value": x, "unit": "TFLOP/s", "n_gpus": 8, "steps": 100, "warmup": 5, "ms_per_step": x,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
        "config": {"workload": "w" * 120, "l2": "l" * 120, "launch": "cuda graph replay", "kernel_path": "default",
                   "parallelism": "replicas only", "also_timed": "per_config: [ms per step, TFLOP/s]"},
        "tokens_per_s": x, "layer_roofline": {"frac_of_measured_burst": x}, "mem_efficiency": {"value": x},
        "activation_bytes": {"saved": 10 ** 9, "scratch": 10 ** 9}, "gpu_launches": 10 ** 6,
        "e2e": {"value": x, "unit": "TFLOP/s", "ms_per_step": x, "h2d_bytes_per_step": 10 ** 9, "d2h_bytes_per_step": 10 ** 9},
        "clocks": {"sm_mhz": x, "sm_mhz_min": x, "sm_max_mhz": x, "reasons": ["sw_power_cap"], "samples": 1000},
        "roofline": {"bound": "tensor", "kernel": "attn_bwd", "achieved": x, "peak": x, "unit": "TFLOP/s", "frac": x, "traffic": x,
                     "kernel_share": x, "kernel_ms": kernel_ms, "timing": "t" * 200},
        "cpu_baseline": {"value": x, "unit": "TFLOP/s", "cores": 16, "kind": "oracle", "sample": "s" * 120, "seconds": x},
        "peaks": {}, "per_config": {"mlp_matmul-512x2048x8192-%d" % i: one for i in range(11)},
    }
    text = json.dumps(bench.contract_line(full))
    assert len(text) < 2800 and "\n" not in text
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline", "dtype",
                "data", "config", "clocks", "e2e", "gpu_launches", "roofline", "cpu_baseline"):
        assert key in line, key
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(line["e2e"])
