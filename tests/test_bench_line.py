"""bench.py prints one line that the end of the output holds whole, with every headline key."""
import json

import bench

HEADLINE = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "roofline", "cpu_baseline", "e2e", "gpu_launches", "clocks")


def _line(steps):
    """As long a line as a run makes: every number at full length, a record per step."""
    x = 0.12345678901234567
    step = {f"field_{k}": x for k in range(18)}
    row = {"workload": "w" * 60, "note": "n" * 120, "ms_per_step": x, "elements_per_s": x * 1e12,
           "lambda_cycle_ends": [x] * 40}
    scan = {"workload": "w" * 60, "batched": dict(row, value=x * 1e10), "one_at_a_time": row, "lams": [[x] * 8] * 32}
    a = bench.parse()
    return {
        "metric": bench.METRIC, "value": x * 1e11, "unit": bench.UNIT, "n_gpus": 1, "steps": steps, "warmup": 5,
        "ms_per_step": x * 1e4, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": bench.config(a, 1), "lanczos_steps_per_s": x,
        "roofline": {"bound": "hbm", "achieved": x, "peak": x, "unit": "GB/s", "frac": x, "traffic": x * 1e12,
                     "kernel": "sigma stage: lists and tables (ms_emit) + gather_kernel (ms_merge)",
                     "peak_kind": "measured copy bandwidth", "ms_per_launch": x, "issue": {"k": [x] * 40},
                     "model": "m" * 300},
        "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 120,
                         "single_thread": {"value": x, "sample": "s" * 120}},
        "e2e": {"value": x, "unit": bench.UNIT, "h2d_bytes_per_step": 16000000, "d2h_bytes_per_step": 16000152,
                "steps": 10, "note": "n" * 200},
        "gpu_launches": 100000, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"]},
        "workloads": {"cfg0": row, "cfg1": row, "cfg2_nd1e5": row, "cfg3_scan": scan, "cfg3_scan_caps_x0.01": scan,
                      "cfg4_rdm": {"ms_per_pass": x, "elements_per_s": x, "note": "n" * 200}},
        "pipe_rates": {f"p{k}": {"ops_per_s": x} for k in range(9)},
        "precision": {"speedup": x, "max_abs_delta_e_comparable": x, "f64": row, "fp32_elements": row},
        "heat_bath_screen": {"runs": [row] * 8},
        "detail": {"timed_steps": [step] * steps, "warmup_steps": [step] * 5},
    }


def test_line_is_short_and_complete(capsys, monkeypatch):
    monkeypatch.setattr("sys.argv", ["bench.py"])
    line = _line(200)
    bench.print_line(line)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) < 2600
    short, full = json.loads(out), json.loads(err)
    assert full == line
    for k in HEADLINE:
        assert k in short
    for k in ("value", "ms_per_step", "config", "clocks", "gpu_launches"):
        assert short[k] == line[k]
    assert short["e2e"]["value"] == line["e2e"]["value"]
    assert short["workloads"]["cfg3_scan"]["value"] > 0
