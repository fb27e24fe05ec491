"""bench.py prints one line that a reader of the last 3000 characters of its output
finds whole, whatever the configurations' records hold."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEADLINE = ["metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
            "scaling", "vs_baseline", "dtype", "data", "config", "roofline", "cpu_baseline", "clocks",
            "gpu_launches"]


def test_line_is_short_and_whole():
    sys.path.insert(0, ROOT)
    import bench

    item = {"ms": 0.31141234, "gflops": 17242.81234, "gbs": 6897.1, "frac": 1.02881234, "passes": 2,
            "tuned": {k: 0 for k in ("radix", "tile", "schedule", "variant", "epilogue", "split_log2")}}
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 14}
    rec = {"workload": "w" * 400, "data": "d" * 120, "ms_per_step": 2.4109953308105467,
           "gflops": 18370.773959611786, "roofline": {"frac": 0.79721234, "achieved": 5344.2}, "clocks": clocks,
           "per_item": {f"16777216 {d} class{i}": item for d in ("fwd", "inv") for i in range(13)}}
    serve = {**rec, "latency_ms": {"p50": 0.51127999999, "p99": 29.341037119}, "achieved_alg_gbs": 3342.331375251816,
             "all_offered_served": True}
    calls = {k: {"host_us": 1.55, "device_us": 2.543, "round_trip_us": 10.688} for k in ("fft_execute", "empty")}
    small = {**rec, "from_c": {"calls": calls, "fft_queue": {"round_trip_us": 9.6, "per_job_us": 6.905}}}
    cufft = {**rec, "per_item": {f"{i}": {**item, "speedup_vs_cufft": 1.25} for i in range(12)}}
    configs = {name: rec for name in bench.SECTION_KEYS.values()}
    configs.update(cfg1_small_call=small, cfg5_serving=serve, cfg5_serving_tc_single_pass=serve,
                   context_cufft=cufft, sar_compression={"error": "RuntimeError: " + "x" * 2000})
    line = {k: 22193.58824329552 for k in HEADLINE}
    line.update(metric=bench.METRIC, data="s" * 125, config={"workload": "w" * 340},
                roofline={"bound": "hbm", "source": "s" * 200}, cpu_baseline={"sample": "s" * 150}, clocks=clocks,
                pct_hbm_roofline=96.6, per_size={f"2^{i}": item for i in range(8, 15)}, autotune_model={"m": "x" * 2400},
                e2e={"value": 924.7090856477855, "unit": "GFLOP/s", "h2d_bytes_per_step": 15032385536,
                     "d2h_bytes_per_step": 15032385536, "steps": 3, "api": "a" * 80, "host_numa": {"x": "y" * 200}},
                configs=configs)
    out = bench.brief_line(line)
    assert len(json.dumps(out)) < 3000
    assert all(out[k] == line[k] for k in HEADLINE)
    assert {k: out["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")} == \
        {k: line["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")}
    assert out["configs"]["cfg5_serving"]["p99_ms"] == 29.341 and out["configs"]["cfg3_multipass"]["frac"] == 0.7972
    assert out["configs"]["context_cufft"]["speedup_vs_cufft_geomean"] == 1.25
    assert out["configs"]["sar_compression"]["error"].startswith("RuntimeError")
    assert bench.brief_line({**line, "e2e": None, "configs": {"skipped": "why"}})["configs"] == {"skipped": "why"}
