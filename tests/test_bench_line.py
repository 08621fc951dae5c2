"""bench.py's result: one short JSON line on stdout that carries the headline, the long sections beside it."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_result_line_is_short_and_whole():
    head = {"metric": bench.METRIC, "value": 1.5e8, "unit": bench.UNIT, "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 700.0, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"model": "m"}, "clocks": {"sm_mhz": 2070.0, "reasons": []}, "gpu_launches": 7,
            "e2e": {"value": 1.4e8, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2}}
    out = dict(head, mixed={"value": 2e8, "search": "x" * 5000}, formulation={"runs": ["y" * 100] * 100})
    details, line = bench.split_result(out)
    assert {k: line[k] for k in head} == head
    assert line["other_paths"]["mixed"] == 2e8
    assert [d["section"] for d in details] == ["mixed", "formulation"]
    assert details[0]["search"] == out["mixed"]["search"] and details[1]["runs"] == out["formulation"]["runs"]
    assert len(json.dumps(line)) < 2000 and "\n" not in json.dumps(line)
    assert bench.split_result(head) == ([], head)
