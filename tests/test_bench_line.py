"""bench.py's printed line is short enough to be read back from the end of a log, whatever the full record
holds, and has the figures it is read for."""
import json

import bench


def _record(extra):
    part = {"events_per_s": 1.23456789012e9, "evals_per_s": 1.0 / 3.0, "what": "x" * extra, "ncu": {"k": ["y" * extra] * 5}}
    line = {"metric": bench.METRIC, "value": 2.1e11 / 3.0, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 0.0475, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "config": {"workload": "w" * 180, "events_per_gpu": 10_000_000, "precision": "p" * 90,
                                            "l2": "l" * 60, "parallelism": "single GPU"},
            "fp64_plain": dict(part, ms_per_eval=0.9), "roofline": {"bound": "issue", "frac": 0.4, "ncu": "z" * extra},
            "e2e": {"value": 5e9 / 7.0, "unit": bench.UNIT, "h2d_bytes_per_step": 120_000_096, "d2h_bytes_per_step": 112,
                    "forms_ms_per_step": {str(i): 1.0 for i in range(extra)}},
            "gpu_launches": 20, "clocks": {"sm_mhz": 2070, "sm_max_mhz": 2070, "reasons": []},
            "oracle_baselines": {"v": ["q" * extra] * 9}}
    for k in bench.FORM_KEYS:
        line[k] = {"workload": "v" * extra, "f32_grad": part, "f64_plain": part}
    for k in ("c5_serving", "c5_serving_poisson"):
        line[k] = {"toys": 4096, "arrival": "Poisson", "fits_per_s": 9000.123456789, "latency_p50_s": 0.2,
                   "latency_p99_s": 0.4, "not_converged": [{"toy": i} for i in range(extra)]}
    return line


def test_line_is_short_and_whole():
    for extra in (1, 10, 3000):
        full = _record(extra)
        text = json.dumps(bench.short_line(full))
        assert len(text) <= bench.MAX_LINE and "\n" not in text
        line = json.loads(text)
        for k in ("metric", "unit", "steps", "warmup", "config", "dtype", "data", "gpu_launches", "clocks", "n_gpus"):
            assert line[k] == full[k]
        assert abs(line["value"] / full["value"] - 1) < 1e-6 and abs(line["e2e"]["value"] / full["e2e"]["value"] - 1) < 1e-6
        assert line["e2e"]["h2d_bytes_per_step"] == 120_000_096 and line["c5_serving"]["fits_per_s"] == 9000.123
        assert line["c3_dalitz_events_per_s"]["f32_grad"] == 1.234568e9
