"""The benchmark's record: one short line on stdout with the headline and what is read beside it, the tables elsewhere."""
import json

import bench


def _record():
    row = {"N": 28672, "K": 8192, "bits": 4, "group": 128, "M": 16, "us": 123.456, "bytes": 132963376, "gbs": 1808.1, "frac": 0.2758}
    out = {"metric": bench.METRIC, "value": 1500.0, "unit": "GB/s", "n_gpus": 1, "ms_per_step": 0.4, "config": {"workload": bench.WORKLOAD},
           "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": []}, "gpu_launches": 680,
           "e2e": {"value": 400.0, "unit": "GB/s", "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 1},
           "roofline": {"bound": "hbm", "achieved": 1500.0, "peak": 6557.8, "cases": [[28672, 8192, 4, 128, 1.0, 16, 1.0, 0.2]] * 300,
                        "cases_columns": "N, K, ..."},
           "prefill_roofline": {"achieved": 1400.0}, "cpu_baseline": {"value": 0.05}}
    out.update({name: [row] * 60 for name in bench.TABLES})
    return out


def test_the_line_is_short_and_the_tables_are_not_lost(capsys, tmp_path):
    out = _record()
    bench.print_record(out, str(tmp_path / "tables.json"))
    shown = capsys.readouterr()
    lines = shown.out.splitlines()
    assert len(lines) == 1 and len(lines[0]) < 4000
    line = json.loads(lines[0])
    for key in ("metric", "value", "unit", "n_gpus", "ms_per_step", "config", "clocks", "gpu_launches", "e2e", "roofline", "cpu_baseline"):
        assert key in line, key
    tables = json.loads((tmp_path / "tables.json").read_text())
    assert {k for t in map(json.loads, shown.err.splitlines()) for k in t} == set(tables)
    assert tables["prefill"] == out["prefill"] and tables["roofline_cases"] == out["roofline"]["cases"]


def test_records_without_tables_pass_through(capsys):
    bench.print_record({"impl": "reference", "value": 1.0})
    assert json.loads(capsys.readouterr().out) == {"impl": "reference", "value": 1.0}
