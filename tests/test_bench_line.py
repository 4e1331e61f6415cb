"""The line bench.py prints: the headline's keys as they are, the legs beside it
cut to rates and times, all of it short."""
import json

import bench


def test_short_line_keeps_the_headline_and_the_rates():
    leg = {"map": "lambda", "value": "hash", "GCells_s": 1.5, "launch_ms": 0.25, "line_GBps": 9.0,
           "profile": "profiles/x.md", "launch_steps": [16] * 64}
    point = {"mode": "batched", "throughput_rps": 5.0, "latency_ms_p99": 0.5, "iterations": 7}
    head = {"metric": "m", "value": 2.5, "unit": "u", "config": {"workload": "w" * 200},
            "clocks": {"sm_mhz": 2070, "reasons": []}, "e2e": {"value": 1.0, "unit": "u"},
            "gpu_launches": 20}
    out = {**head,
           "compare": {**{f"leg{i}": dict(leg) for i in range(24)}, "speedup": 6.0,
                       "level_sweep": {f"r{r}": {"lambda_us": 2.0, "bbox_us": 3.0, "speedup": 1.5}
                                       for r in range(8, 17)},
                       "write_sweep_best": {"protocol": "p", "best_per_level": {
                           f"{t}_r{r}": {"lambda_us": 2.0, "bbox_us": 3.0, "lambda_rho": 8}
                           for t in ("u8", "f32") for r in range(8, 17)}},
                       "compact": {"rho": 64, "order": "interleaved", "ca": dict(leg)}},
           "serving": {"offered": {"batched": dict(point)},
                       "saturation": {"p99_bound_ms": 5.0, "rates_rps": [1.0] * 11, "modes": {
                           "batched": {"max_sustained_rps": 4.0, "points": [dict(point)] * 40}}}},
           "e2e_paths": {"copy": {"value": 1.0, "ms_per_step": 2.0, "path": "p" * 300}}}
    before = json.dumps(out)
    line = bench.short_line(out)
    assert json.dumps(out) == before                   # what --report writes is not cut
    assert {k: line[k] for k in head} == head
    assert line["compare"]["leg3"] == {"GCells_s": 1.5, "launch_ms": 0.25}
    assert line["compare"]["speedup"] == 6.0
    assert line["compare"]["compact"] == {"rho": 64, "ca": {"GCells_s": 1.5, "launch_ms": 0.25}}
    assert line["compare"]["level_sweep_us"]["r16"] == [2.0, 3.0]
    assert line["compare"]["write_sweep_best_us"]["f32_r8"] == [2.0, 3.0]
    assert line["serving"]["offered"]["batched"] == {"throughput_rps": 5.0, "latency_ms_p99": 0.5}
    assert line["serving"]["saturation"]["modes"]["batched"] == {"max_sustained_rps": 4.0}
    assert line["e2e_paths"]["copy"] == {"value": 1.0, "ms_per_step": 2.0}
    assert len(json.dumps(line)) < 8000 < len(before)


def test_a_quick_result_is_printed_as_it_is():
    out = {"metric": "m", "value": 1.0, "roofline": {"frac": 0.5, "kernel": "k"}}
    assert bench.short_line(out) == out
