"""bench.py's result line holds the headline alone: the tables of the other
workloads (30 KB) go to stderr, so that the line, `value` first of all, survives a
reader that keeps a few KB of stdout."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402


def test_result_line_is_the_headline_alone():
    big = [{"T": t, "errors": {k: 1.0 / 3.0 for k in "SvKxu"}} for t in range(100)]
    head = {"metric": bench.METRIC, "value": 3.4e9, "unit": bench.UNIT, "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 0.3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": bench.workload_config(1000000),
            "e2e": {"value": 9e8, "unit": bench.UNIT, "h2d_bytes_per_step": 8000232,
                    "d2h_bytes_per_step": 136000096}, "clocks": {"sm_mhz": 2070.0},
            "gpu_launches": 200}
    line = dict(head, **{k: big for k in bench.DETAILS})
    got, details = bench.split_line(line)
    assert {k: got[k] for k in head} == head
    assert set(got) - set(head) == {"details"}
    assert details == {k: big for k in bench.DETAILS}
    assert len(json.dumps(got)) < 3000 < len(json.dumps(line))
