"""bench.py prints one short JSON line on stdout: every key of its contract, however many
workloads the run measures beside the metric, whose figures go elsewhere whole."""
import json

import bench


def report():
    legs = {f"leg{i}": {"workload": "w" * 200, "forms": [{"iters_per_s": 1.0 / 3.0}] * 20}
            for i in range(12)}
    roof = {"bound": "tensor", "achieved": 1.0 / 3.0, "peak": 1967.6, "unit": "TFLOP/s", "frac": 1.0 / 3.0,
            "traffic": 14706944.0, "kernel": "tc_loop_kernel (BF16)", "kernel_ms": 1.0 / 3.0,
            "us_per_pair": 1.0 / 3.0, "flops_note": "n" * 400, "executed_note": "n" * 400,
            "per_pass_kernels": {"passes_ms": [0.1] * 4}, "traffic_unit": "bytes per launch"}
    return {"metric": bench.METRIC, "value": 1.0 / 3.0, "unit": bench.UNIT, "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 1.0 / 3.0, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "bf16", "data": "synthetic", "config": bench.bench_config(1024),
            "run": {"precision": "BF16", "parallelism": "replicas1", "steps_timed": "JKO steps 6..25",
                    "headline_rule": "fastest tensor-core form with " + "r" * 100 + " < 1e-3"},
            "jko_steps_per_s": 1.0 / 3.0, "iters_per_step": [200] * 20, "forms": legs["leg0"],
            "wall_s": 1.0 / 3.0, "roofline": roof,
            "cpu_baseline": {"value": 1.0 / 3.0, "unit": bench.UNIT, "cores": 16, "kind": "oracle",
                             "sample": "s" * 100},
            "accuracy_vs_oracle": legs["leg1"],
            "e2e": {"value": 1.0 / 3.0, "unit": bench.UNIT, "h2d_bytes_per_step": 4194304,
                    "d2h_bytes_per_step": 4194304},
            "gpu_launches": 1000, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []}, **legs}


def test_line_is_short_and_holds_the_contract():
    line = report()
    short, rest = bench.split_report(line)
    text = json.dumps(short)
    assert len(text) < 2600 and "\n" not in text
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                "scaling", "vs_baseline", "dtype", "data", "config", "e2e", "gpu_launches", "clocks",
                "roofline", "cpu_baseline"):
        assert key in short, key
    assert {**short, **rest} == line          # nothing is lost between the two
