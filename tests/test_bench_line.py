"""The line bench.py prints stays short enough to be read from the end of its output."""
import json
import os
import sys

from conftest import ROOT

sys.path.insert(0, ROOT)
import bench  # noqa: E402


def test_the_line_is_short_and_the_rest_is_detail():
    long = {f"k{i}": [0.1234567] * 40 for i in range(30)}
    line = {key: 1.25 for key in bench.LINE_KEYS}
    line.update(metric=bench.METRIC, unit=bench.UNIT, scaling="weak", dtype="bf16", data="synthetic",
                config={"workload": "w" * 90, "search": "s" * 90, "T": 32, "l2": "l" * 90, "precision": "p" * 30},
                e2e={"value": 1.0, "unit": bench.UNIT, "h2d_bytes_per_step": 1, "d2h_bytes_per_step": 2},
                clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
                roofline=dict({key: 1.0 for key in bench.ROOFLINE_KEYS}, per_query_model=long, tensor=long),
                cpu_baseline={"value": 1.0, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "x" * 90, "fp32_loop": long},
                paths=long, configs=long, serving=long, accuracy=long)
    short, detail = bench.contract_line(line)
    assert len(json.dumps(short)) < 2500
    assert set(short) == set(bench.LINE_KEYS)
    assert short["value"] == line["value"] and short["e2e"] == line["e2e"] and short["config"] == line["config"]
    assert short["cpu_baseline"]["value"] == 1.0 and short["roofline"]["frac"] == 1.0
    assert detail == {key: line[key] for key in ("paths", "configs", "serving", "accuracy", "roofline", "cpu_baseline")}
