"""The result line of bench.py stays short enough for a reader that keeps the
last 3000 characters of the output, whatever lists the record holds, and loses
no key that says what was measured."""
import json

import bench


def _record():
    curve = {p: {"per_step": [1.234567890123e-3] * 57, "after_step_1": 1e-3, "final_336h": 4.92571077588023e-07,
                 "final_337h": 4.983008243887112e-07, "max": 4.983008243887112e-07, "nonfinite_final": 0}
             for p in ("fp32", "bf16", "fp8mlp")}
    figures = {n: {**{k: 123.45678901234567 for k in ks}, "workload": "x" * 200, "by_lead": [1.0] * 50}
               for n, ks in bench.SECTION_FIGURES.items()}
    kernels = {k: 1.2345678901234567 for k in ("ln1", "qkv", "attn", "proj", "ln2", "fc1", "fc2")}
    return {"metric": bench.METRIC, "value": 48.0354648557789, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 20.817951965332032, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "bf16", "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "batch_per_gpu": 1, "blocks": 8, "parallelism": "single GPU",
                       "l2": "working set larger than L2 (latent 448 MB fp32, activations ~2 GB bf16)"},
            "gpu_launches": 820, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 5},
            "roofline": {"bound": "hbm", "kernel": "attn", "achieved": 825.58877, "peak": 6677.2, "unit": "GB/s",
                         "frac": 0.1236, "traffic": None, "peak_source": "measured HBM copy bandwidth",
                         "kernels_ms_per_step": kernels, "gemm_tflops": kernels, "attn_halo": {"plan": "x" * 300}},
            "e2e": {"value": 47.4, "unit": bench.UNIT, "h2d_bytes_per_step": 447897600, "d2h_bytes_per_step": 447897600,
                    "call": "wm_forecast_host_many(lead 6 h, K forecasts)", "clocks": {"samples": 9},
                    "single_call": {"value": 40.4}},
            "autotune": ["  candidate " + "x" * 80] * 150, "rollout_error_vs_oracle": curve,
            "cpu_baseline": {"value": 1.6e-3, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "x" * 250,
                             "seconds_per_forecast": 618.3, "small_latent": {"block_s_1_thread": 1.0},
                             "rollout_337h_small": {"seconds": 1.0}}, **figures}


def test_line_is_short_and_complete():
    record = _record()
    assert len(json.dumps(record)) > 10000
    text = json.dumps(bench.result_line(record))
    assert "\n" not in text and len(text) < 2900, len(text)
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks"):
        assert line[key] == record[key]
    for key in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"):
        assert line["e2e"][key] == record["e2e"][key]
    for key in ("bound", "kernel", "achieved", "peak", "unit", "frac"):
        assert line["roofline"][key] == record["roofline"][key]
    for prec in ("fp32", "bf16", "fp8mlp"):
        assert line["rollout_error_vs_oracle"][prec]["final_336h"] == 4.92571077588023e-07
