"""The line that the benchmark prints is short enough to be read whole from a bounded tail of the
output, whatever was measured beside it, and keeps the contract's keys."""

import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def _full():
    """A result with every part present and numbers of full length."""
    x, long = 12345.678901234567, "w" * 200
    e2e = {"value": x, "unit": "events/s", "host_threads": 3, "h2d_bytes_per_step": 10**9,
           "d2h_bytes_per_step": 10**9}
    stages = dict.fromkeys(("load", "doublets", "connect", "ntuplets", "fit"), 123.4567)
    kernels = {f"k_kernel_with_a_name_{i}": x for i in range(20)}
    form = {"value": x, "ms_per_step": x, "p99_ms_per_step": x, "stages_ms": stages, "e2e": e2e,
            "kernels_ms": kernels}
    physics = {"efficiency": 0.98454977194265, "fake_rate": x, "duplicate_rate": x,
               "n_fake": 10**6, "n_ntuplets": 10**7, "events": 128}
    rate = {"p50_ms": 123.45678, "p99_ms": 1234.5678, "workload": long,
            **{f"number_{i}": x for i in range(20)}}
    serving = [dict(rate, offered_events_per_s=r)
               for r in (200.0, 1000.0, 2000.0, 4000.0, 6000.0, 8000.0, 10000.0, 12000.0)]
    part = {"ms_per_step": x, "workload": long, "events_per_step": 64}
    latency = dict.fromkeys(("config1_barrel50", "pu50_single", "pu200_single"),
                            {"p50_ms": x, "p99_ms": x, "path": long})
    return {"metric": bench.METRIC, "value": x, "unit": "events/s", "n_gpus": 1, "steps": 60,
            "warmup": 3, "ms_per_step": x, "p99_ms_per_step": x, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": bench.WORKLOAD, "events_per_step": 64, "form": "plain",
                       "phi_bins": 2048, "blocks_per_sm": 8, "search_blocks_per_sm": 8,
                       "tuning": "autotuned (measured)",
                       "l2": "flushed before every step (256 MB write, outside the events)",
                       "parallelism": "replicas x1"},
            "e2e": e2e, "stages_ms": stages, "kernels_ms": kernels, "gated": form,
            "roofline": {"bound": "hbm", "kernel": "k_connect", "achieved": x, "peak": x,
                         "unit": "GB/s", "frac": x, "traffic": 10**10, "peak_src": "measured",
                         "algorithmic_bytes": 10**10, "launch_ms": x, "issue_active_pct": x,
                         "steps": kernels, "issue": kernels},
            "physics": {"plain": physics, "gated": physics},
            "counts_per_step": dict.fromkeys("abcdefg", 10**9),
            "batch_workload": {"plain": dict(part, value=x), "gated": dict(part, value=x)},
            "latency": dict(latency, batches={"value": x}), "gap_pairs": part, "fishbone": part,
            "vertexing": part, "broken_line": part, "raw_input": part,
            "autotune": {f"{i}x8x8": x for i in range(60)},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 3},
            "gpu_launches": 1320,
            "serving": {"plain": serving, "gated": serving, "instances": serving[:3]},
            "cpu_baseline": {"value": x, "unit": "events/s", "cores": 16, "kind": "oracle",
                             "sample": long[:90], "host_cores": 16, "one_thread": rate}}


def test_line_is_short_and_complete():
    full = _full()
    assert len(json.dumps(full)) > 10000
    line = bench.short_line(full, "bench_details.json")
    assert len(json.dumps(line)) <= bench.LINE_BYTES
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
              "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
              "clocks", "gpu_launches", "roofline", "gated", "efficiency", "details"):
        assert k in line, k
    assert line["value"] == full["value"] and line["e2e"] == full["e2e"]
    assert line["config"] == full["config"] and line["clocks"] == full["clocks"]


def test_line_without_the_optional_parts():
    full = _full()
    for k in ("serving", "cpu_baseline"):
        del full[k]
    full.update(latency=None, e2e=None, physics={"plain": None, "gated": None})
    full["gated"]["e2e"] = None
    line = bench.short_line(full, "d.json")
    assert "vs_baseline" in line and "efficiency" not in line and line["value"] == full["value"]
