"""The benchmark's output line: complete, and short enough to be read from an output's last characters."""
import json

import bench

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline")


def _roof(name):
    return bench.roof(name, 45_863_262_208, [6.9123, 7.1456, 6.8123] * 8, 6547.8, "measured")


def test_the_line_is_short_and_keeps_what_it_has_to_say():
    rec = {"workload": "w" * 160, "steps": 400, "value": 123456.7, "unit": bench.UNIT, "ms_per_step": 0.01234,
           "step_frac_of_peak": 1.0123, "step_frac_of_nominal": 0.8123, "l2": "l" * 80,
           "roofline_ctc": _roof("ctc_rows_tma"), "roofline_verify": _roof("verify_rows_direct"),
           "cpu_baseline": {"value": 2.42, "sample": "s" * 150}}
    line = {k: 1 for k in CONTRACT}
    line.update(metric=bench.METRIC, unit=bench.UNIT, value=71234.5, data="synthetic", dtype="f32",
                config={"workload": "w" * 170, "calls_per_step": "c" * 90, "l2": "l" * 110, "parallelism": "p" * 60},
                clocks={"sm_mhz": 1620.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"], "note": "n" * 120},
                e2e={"value": 1234.5, "unit": bench.UNIT, "h2d_bytes_per_step": 10 ** 11, "d2h_bytes_per_step": 10 ** 5,
                     "note": "n" * 300},
                roofline=_roof("verify_rows_direct"), roofline_ctc=_roof("ctc_rows_tma"),
                roofline_verify=_roof("verify_rows_direct"), decisions={"gate_accept_frac": 0.1},
                next_rows={"x": "y" * 2500}, cpu_baseline=dict(rec["cpu_baseline"], kind="oracle", cores=16),
                per_config={name: rec for name, *_ in bench.PER_CONFIG})
    text = bench.short_line(line)
    assert len(text) <= bench.LINE_LIMIT and "\n" not in text
    got = json.loads(text)
    assert all(k in got for k in CONTRACT)
    assert got["value"] == 71234.5 and got["roofline"]["frac"] == line["roofline"]["frac"]
    assert set(got["per_config"]) == set(line["per_config"]) and "cpu_baseline" in got
