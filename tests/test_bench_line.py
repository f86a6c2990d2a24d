"""The line bench.py prints: one JSON object, short enough for a log that keeps only the end of a
run's output, whatever the sweeps hold; the full record keeps every row."""
import json

import bench
from paper_2505_19645_b200 import workloads as wl


def _record():
    row = {"B": 512, "gamma": 5, "T": 3072, "us": 4222.94, "roof_frac": 0.82, "n_active": 256}
    f = 1234.5678901234567
    return {
        "metric": "moe_verify_layer_tokens_per_s", "value": 41361.303764446595, "unit": "tokens/s", "n_gpus": 8,
        "steps": 200, "warmup": 10, "ms_per_step": 3.0946800112724304, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic (seeded)",
        "config": {"workload": "qwen1.5-moe-a2.7b-dense-shaped MoE FFN layer, B=1024, gamma=15 (T=16384 tokens)",
                   "config": "qwen1.5-moe-a2.7b", "B": 1024, "gamma": 15, "tokens": 16384, "zipf": 1.25,
                   "shape": wl.dense_contrast(wl.CONFIGS["qwen1.5-moe-a2.7b"]).as_dict(),
                   "l2": "512 MiB buffer written between timed iterations", "parallelism": "replicas only"},
        "roofline": {"bound": "tensor", "achieved": f, "peak": 6547.8, "unit": "TFLOP/s", "frac": f,
                     "traffic": 123456789012, "kernel": "layer_small_kernel (whole layer in one launch)",
                     "kernel_ms": f, "algorithmic_bytes": 123456789012, "peak_source": "measured"},
        "layer_roofline": dict({k: f for k in ("roof_ms", "frac", "frac_of_nominal", "n_active_expected",
                                               "frac_sustained_tensor_peak", "t_exp", "t_exp_expected",
                                               "median_ms", "min_ms")},
                               bound="tensor", n_active=256, t_thres=12345, beyond_t_thres=False,
                               bytes=123456789012, flops=1234567890123456,
                               peaks={"hbm_gbs": 6547.8, "bf16_tflops": 1610.2, "bf16_tflops_sustained": 1353.0,
                                      "source": "earlier measurement on this GPU type",
                                      "nominal_hbm_gbs": 7700.0, "nominal_bf16_tflops": 2250.0}),
        "cpu_baseline": {"value": f, "unit": "tokens/s", "cores": 128, "kind": "oracle",
                         "sample": "512 seeded token rows of the T=16384 batch, 200 passes, 10.0 s"},
        "e2e": {"value": f, "unit": "tokens/s", "h2d_bytes_per_step": 123456789, "d2h_bytes_per_step": 123456789},
        "gpu_launches": 1600, "layer_us": f,
        "clocks": {"sm_mhz": 1770.0, "sm_min_mhz": 1215.0, "sm_max_mhz": 1965.0, "samples": 1234,
                   "reasons": ["sw_power_cap", "hw_slowdown", "sw_thermal_slowdown"]},
        "small_batch": {"T1_layer_us": f, "T1_e2e_us": f, "T1_e2e_h2d_bytes": 14336,
                        "host_us_per_call": {"T1": f, "T16384": f},
                        "host_us_per_call_c_abi": {"T1": f, "T16384": f}, "host_us_per_call_how": "x" * 300},
        "sweeps": {key: {"rows": [dict(row, roof_frac=0.02 * i) for i in range(40)]}
                   for key, _, _ in bench.ALL_SWEEPS},
    }


def test_the_line_is_short_and_keeps_the_contract_keys():
    record = _record()
    text = bench.result_line(record)
    assert len(text) <= bench.LINE_MAX < 3000 and "\n" not in text
    line = json.loads(text)
    assert set(line) == set(record)
    for key, want in record.items():
        if key not in ("sweeps", "small_batch"):
            assert line[key] == bench.rounded(want), key
    assert abs(line["value"] / record["value"] - 1) < 1e-6
    assert line["sweeps"] == {key: [40, 5] for key, _, _ in bench.ALL_SWEEPS}
    # the record itself is left as it was
    assert len(record["sweeps"]["tiny"]["rows"]) == 40 and "host_us_per_call_how" in record["small_batch"]
