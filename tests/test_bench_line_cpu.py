"""The bench's JSON line: the headline keys whole, the side sections as their times, a few kilobytes in all."""
import json


def _out():
    curve = {"seconds": 0.1, "ms_per_iteration": 1.234567, "gap_curve": [0.1] * 30, "rollout": "bf16", "launch_variants": {"a": 1}}
    many = {f"variant {i}": dict(curve) for i in range(14)}
    out = {"metric": "m", "value": 5.0, "unit": "u", "n_gpus": 1, "steps": 10, "warmup": 3, "ms_per_step": 8.0,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
           "config": {"workload": "w" * 300}, "roofline": {"frac": 0.4}, "clocks": {"sm_mhz": 2070.0}, "gpu_launches": 90,
           "e2e": {"value": 4.0, "unit": "u", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2}, "cpu_baseline": {"value": 1.0}}
    out.update(time_to_gap=dict(many, target_gap=0.04), time_to_gap_pushing=dict(many), batched=dict(curve),
               manip_scale={"ibp_ms": 18.5, "rollout_bf16_ms": 2.5, "iteration": {"fp32_intervals": dict(curve)}},
               paper_bounding=dict(many), heuristics={"alpha": dict(many), "workload": "x"}, cem_search=None,
               tiny_latency={"us_per_iteration_graph": 87.5, "status": 0},
               precision_lines={"fp32": {"ms_per_step": 113.04669, "kernel_ms": {"rollout": 111.7}, "roofline": {"frac": 0.6}}})
    return out


def test_line_keeps_the_headline_and_is_short():
    import bench
    out = _out()
    line, details = bench.split_line(out)
    text = json.dumps(line)
    assert len(text) < 6000 < len(json.dumps(out)) and "\\n" not in text
    for key in out:
        assert (details if key in bench.SIDE_SECTIONS else line)[key] == out[key]
    side = line["side_ms"]
    assert side["precision_lines"] == {"fp32": 113.0} and side["batched"] == 1.235 and side["tiny_latency"] == 87.5
    assert side["time_to_gap"]["variant 3"] == 1.235 and "cem_search" not in side
    assert side["manip_scale"] == {"ibp_ms": 18.5, "rollout_bf16_ms": 2.5, "iteration": {"fp32_intervals": 1.235}}
