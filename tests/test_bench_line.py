"""The line bench.py prints: short enough for a reader that keeps the last 4 kB of a run's output, with every key of the
measurement; the sections in full go to stderr."""
import json

import bench


def test_the_printed_line_is_short_and_complete():
    big = {f"k{i}": 1.2345678901234567 for i in range(200)}
    line = {"metric": bench.METRIC, "value": 75.594, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 13.2, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": bench.workload_name(512, 512), "nodes": 263169, "parallelism": "single GPU"},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "e2e": {"value": 70.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
            "gpu_launches": 50000, "launches_per_step": 2500.0, "iters_per_step_mean": 14.0, "iters_per_step_max": 19,
            "amg_levels": {"M": [263169, 30000, 500], "H": [263169, 30000, 500]},
            "cpu_baseline": {"value": 0.6, "unit": bench.UNIT, "cores": 1, "kind": "oracle", "error_vs_oracle_per_step": big}}
    for name in list(bench.SECTION_KEYS) + list(bench.DETAIL_ONLY):
        line.setdefault(name, dict(big))
    line["mixed"].update(value=203.6, ms_per_step=4.9)
    form = {"steps_per_s": 192.93246767488424, "ms_per_step": 5.183160781860352, "iters_per_step_mean": 11.1375}
    line["learned"].update({p: {k: dict(form) for k in ("previous_state", "learned", "linear_extrapolation",
                                                        "quadratic_extrapolation")} for p in ("fp64", "mixed")})
    out = bench.stdout_line(line)
    text = json.dumps(out)
    assert len(text) < 4000 and "\n" not in text
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
                "dtype", "data", "config", "clocks", "e2e", "gpu_launches"):
        assert out[key] == line[key]
    assert out["mixed"] == {"value": 203.6, "ms_per_step": 4.9} and out["cpu_baseline"]["value"] == 0.6
    assert bench.stdout_line(dict(line, mixed=None, batch=None))["mixed"] is None
