"""bench.py's line on stdout stays short however much was timed: a log's tail of a few thousand characters has to hold all of it."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

LIMIT = 4000
NUMBER = 1234.5678901234567   # as long as a float prints


def test_headline_holds_the_contract_and_stays_short():
    import bench
    calls = {c: NUMBER for c in bench.CALLS}
    clocks = {"sm_mhz": NUMBER, "sm_max_mhz": 1965, "reasons": ["sw_power_cap", "hw_thermal_slowdown"], "samples": 1000, "power_w_max": NUMBER}
    roofline = {k: NUMBER for k in bench.HEADLINE_ROOFLINE_KEYS + ("frac_of_burst", "frac_of_nominal_2250")}
    roofline.update(kernel="grouped_gemm_kernel[gateup_swiglu]", traffic_source="x" * 80)
    summary = dict(workload="fine_grained", ms_per_step=NUMBER, layer_tflops=NUMBER, per_call_ms=calls, per_call_tflops=calls,
                   roofline=roofline, clocks=clocks, mxfp8={c: calls for c in calls}, fp8_step=calls)
    line = {k: NUMBER for k in bench.HEADLINE_KEYS}
    line.update(metric=bench.METRIC, unit=bench.UNIT, data="synthetic", clocks=clocks, roofline=roofline, detail=summary,
                mxfp8=summary["mxfp8"], other_configs=[dict(summary, workload=f"workload_{i}") for i in range(5)],
                config={k: "x" * 60 for k in ("workload", "T", "H", "I", "E", "K", "routing", "parallelism", "timed_seconds", "l2")},
                peaks={k: NUMBER for k in ("kind", "hbm_gbs", "bf16_tflops", "bf16_tflops_sustained", "nominal_bf16_tflops", "nominal_hbm_gbs")},
                e2e={"value": NUMBER, "unit": bench.UNIT, "h2d_bytes_per_step": 10 ** 9, "d2h_bytes_per_step": 10 ** 9, "ms_per_step": NUMBER,
                     "results_equal_device_resident_step": True, "note": "x" * 400},
                cpu_baseline={"value": NUMBER, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "x" * 150, "seconds": NUMBER})
    assert len(json.dumps(line)) > 2 * LIMIT
    out = bench.headline(line)
    text = json.dumps(out)
    assert len(text) <= LIMIT, len(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                "dtype", "data", "config", "clocks", "gpu_launches"):
        assert out[key] == line[key]
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(out["e2e"])
    assert out["roofline"]["achieved"] == NUMBER and len(out["other_configs"]) == 5
