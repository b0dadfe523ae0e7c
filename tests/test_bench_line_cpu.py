"""The result line of bench.py stays short whatever the run measured; what is taken out of it is kept beside it."""
import json

import bench


def test_long_parts_leave_the_result_line():
    line = {"metric": bench.METRIC, "value": 1.5, "unit": "GB/s", "n_gpus": 1, "config": {"workload": "w" * 300},
            "roofline": {"kernel": "k", "frac": 0.9, "configs": [{"line": "x" * 80, "ms": 0.1}] * 40},
            "transforms": [{"transform": "t" * 60, "ms": 0.1}] * 7, "ops": [{"op": "o" * 80, "ms": 0.2}] * 40,
            "cpu_baseline": {"value": 1.0, "configs": [{"what": "y" * 80}] * 6}, "e2e": {"value": 2.0}, "clocks": {"sm_mhz": 1965}}
    whole = json.loads(json.dumps(line))
    record, detail = bench.split_record(line)
    assert len(json.dumps(record)) < 2048
    assert {"metric", "value", "unit", "n_gpus", "config", "roofline", "cpu_baseline", "e2e", "clocks"} == set(record)
    assert record["roofline"] == {"kernel": "k", "frac": 0.9} and record["cpu_baseline"] == {"value": 1.0}
    assert detail["ops"] == whole["ops"] and detail["transforms"] == whole["transforms"]
    assert detail["roofline_configs"] == whole["roofline"]["configs"] and detail["cpu_baseline_configs"] == whole["cpu_baseline"]["configs"]
    assert line == whole, "the record taken apart is left as it was"
