"""The bench's result is one short line on standard output; the long tables go to standard error."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_the_line_is_short_and_nothing_is_lost(capsys):
    # a line with what a run reports, numbers at full length
    x = 0.1 + 1.0 / 3.0
    phase = {"ms_per_launch": x, "launches": 20, "algo_GBps": x * 1e4}
    line = {"metric": bench.METRIC, "value": x, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5, "ms_per_step": x,
            "config": {"workload": "cosmo_512p_1024m_2048r", **{f"key_{i}": "some words on the run" for i in range(12)}},
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 7}, "gpu_launches": 192,
            "phases": {f"phase_{i}": phase for i in range(8)}, "e2e": {"value": x, "returned": "words " * 30},
            "cpu_baseline": {"value": x, "sample": "words " * 40},
            "next_rows": {"table": [x] * 400}, "precision": {"table": [x] * 400}, "learned": {"table": [x] * 400}}
    bench.report(line)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and err.count("\n") == 1
    assert len(out) < 4096
    short, details = json.loads(out), json.loads(err)
    assert set(short).isdisjoint(bench.DETAILS) and {**short, **{k: details[k] for k in bench.DETAILS}} == line


def test_a_run_without_tables_prints_no_second_line(capsys):
    bench.report({"value": 1.0, "config": {"workload": "w"}, "next_rows": None})
    out, err = capsys.readouterr()
    assert json.loads(out) == {"value": 1.0, "config": {"workload": "w"}} and err == ""
