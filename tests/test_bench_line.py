"""The benchmark's stdout line stays short whatever the record holds, and keeps the keys its readers need."""
import json

import bench


def _record(blocks):
    long = "x" * 400
    record = {"metric": bench.METRIC, "value": 646.123456789012, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
              "ms_per_step": 0.37412345678901, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
              "dtype": "int8", "data": "synthetic", "wall_s_timed_region": 1.23456789012345, "gpu_launches": 3000,
              "config": {"workload": bench.workload_name(5), "layers": 10, "launch": "CUDA graph replay",
                         "l2": "flushed before every replay (256 MiB memset outside the replay's event pair)",
                         "parallelism": "single GPU"},
              "clocks": {"sm_mhz": 1965, "sm_max_mhz": 1965, "reasons": ["sw_power_cap"], "samples": 200},
              "timing": {"note": long}, "us_per_layer": [1.23456789012345] * 10}
    if blocks:
        figures = {"value": 646.123456789012, "unit": "TOPS", "us_per_step": 374.123456789012, "note": long,
                   "kernels": {k: {"us_per_step": 1.0, "note": long} for k in bench.KERNELS}}
        record.update(
            warm=figures, sustained=figures, contraction={"note": long}, nhwc_input=figures, w4_weights=figures,
            layers_on_three_streams=figures, per_config={f"cfg{i}": dict(figures) for i in range(1, 6)},
            full_quant={"y_per_tile": figures, "y_per_row_column": {"error": long}},
            parity={"ok": True, "worst_rel_err": 2.450367866059461e-06, "against": long},
            cpu_baseline={"value": 0.29, "unit": "TOPS", "cores": 16, "kind": "oracle", "sample": long},
            roofline={"bound": "hbm", "kernel": bench.KERNELS[1], "achieved": 2633.123456789, "peak": 6549.8, "unit": "GB/s",
                      "frac": 0.40212345678, "traffic": 39228851, "launches_per_step": 10, "note": long, "all_kernels": figures},
            e2e={"value": 103.80189552647907, "unit": "TOPS", "h2d_bytes_per_step": 44564480, "d2h_bytes_per_step": 104857600,
                 "steps": 20, "api": long, "serial": figures})
    else:
        record.update(parity=None, e2e=None, cpu_baseline=None, per_config=None, full_quant=None, roofline=None)
    return record


def test_line_is_short_and_complete():
    record = _record(True)
    assert len(json.dumps(record)) > 2 * bench.LINE_LIMIT
    text = bench.printed_line(record)
    assert len(text) <= bench.LINE_LIMIT and "\n" not in text
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "clocks", "gpu_launches"):
        assert line[key] == record[key], key
    assert line["e2e"]["value"] == record["e2e"]["value"]
    assert line["e2e"]["h2d_bytes_per_step"] == 44564480 and line["e2e"]["d2h_bytes_per_step"] == 104857600


def test_line_of_a_run_without_the_extra_legs():
    record = _record(False)
    line = json.loads(bench.printed_line(record))
    assert line["value"] == record["value"] and line["e2e"] is None and "values" not in line
