"""The benchmark's printed line: one short JSON line with the contract's fields, the long sections
in the detail file."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402

CONTRACT = ["metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step",
            "higher_is_better", "scaling", "vs_baseline", "dtype", "data", "config", "e2e",
            "gpu_launches", "clocks"]


def record():
    x = 123456789.123456789
    rate = {"value": x, "ms": x, "unit": bench.UNIT, "wall_s": x, "box_evals": 10 ** 11}
    long = {"cell-%d" % i: {"ms": x, "note": "a sub-report of a run " * 3} for i in range(80)}
    r = {k: x for k in CONTRACT}
    r.update({
        "metric": bench.METRIC, "unit": bench.UNIT, "data": "synthetic", "scaling": "weak",
        "dtype": "f32 (float pairs, then f64, on the error band)", "higher_is_better": True,
        "config": bench.config_dict(1, "binary32 intervals from the full level-6 grid; the error "
                                       "band re-decided at the last level"),
        "e2e": {"value": x, "unit": bench.UNIT, "h2d_bytes_per_step": 10 ** 7,
                "d2h_bytes_per_step": 10 ** 9, "steps": 5, "ms_each": [x] * 5, "what": "w" * 300},
        "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "samples": 10, "power_w_max": x,
                   "reasons": ["sw_power_cap"]},
        "fp64": {"value": x, "ms_per_step": x, "steps": 2, "roofline": long},
        "roofline": {"kernel": "leaf_fp32", "bound": "alu", "algorithmic_madds_per_s": x,
                     "algorithmic_ops_over_peak": x, "note": "n" * 80, "traffic": x,
                     "traffic_unit": "bytes per launch (DRAM read + write)", "launches": 25,
                     "avg_launch_ms": x, "madds_per_launch": x,
                     "time_share": {"kind%d" % i: x for i in range(12)},
                     "peak_basis": {"sms": 152, "sm_mhz": 2070.0, "lanes_per_sm": 128}},
        "cpu_baseline": {"value": x, "unit": bench.UNIT, "cores": 1, "kind": "oracle",
                         "sample": "s" * 250},
        "every_level_recheck": {"ms_median": x, "value": x, "what": "w" * 90},
        "enclosure_ms": {"median": x, "min": x, "max": x, "cold": {"note": "n" * 90}},
        "batch": {"fp32": rate, "fp64": rate, "fp32_recheck_last": rate,
                  "fp32_equals_fp64": True, "fp32_recheck_last_equals_fp64": True, "more": long},
        "dense_level": {"fp32": rate, "fp64": rate, "fp32_equals_fp64": True,
                        "tensor_core": {"exact_fp32": rate, "more": long}},
    })
    for k in bench.DETAIL:
        r.setdefault(k, long)
    return r


def test_the_line_is_short_and_the_file_has_everything(tmp_path, capsys):
    path = str(tmp_path / "detail.json")
    r = record()
    assert len(json.dumps(r)) > 20000
    bench.print_record(r, path)
    out = capsys.readouterr().out.splitlines()
    assert len(out) == 1 and len(out[0]) <= bench.MAX_LINE
    line = json.loads(out[0])
    assert [k for k in CONTRACT if k not in line] == []
    for k in ("value", "ms_per_step", "config", "clocks", "gpu_launches"):
        assert line[k] == r[k]
    assert {k: line["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")} \
        == {k: r["e2e"][k] for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")}
    assert line["roofline"]["kernel"] == "leaf_fp32" and line["brief"]["batch"]["same"] is True
    assert json.load(open(path)) == r and line["detail"] == "detail.json"


def test_without_sub_reports_or_a_place_for_the_file(tmp_path, capsys):
    r = {k: v for k, v in record().items() if k not in bench.DETAIL}
    r["cpu_baseline"] = None
    for path in ("", str(tmp_path / "no" / "such" / "folder.json")):
        bench.print_record(r, path)
        line = json.loads(capsys.readouterr().out)
        assert "detail" not in line and "brief" not in line and line["value"] == r["value"]


def test_a_long_line_loses_only_what_the_contract_does_not_name(capsys):
    r = record()
    r["cpu_baseline"]["sample"] = "s" * 4000
    bench.print_record(r, "")
    line = json.loads(capsys.readouterr().out)
    assert [k for k in CONTRACT if k not in line] == [] and "cpu_baseline" not in line
