"""The benchmark's one line on standard output holds the contract's keys and no secondary leg; the legs
go to standard error, every one of them."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402


def test_legs_are_no_part_of_the_line():
    head = {"metric": bench.METRIC, "value": 1.0, "e2e": {"value": 1.0}, "gpu_launches": 4, "clocks": {}, "parity": {}}
    legs = {k: {"results": "x" * 4000} for k in bench.LEGS}
    line, rest = bench.split_line({**head, **legs})
    assert line == head and rest == {"legs": legs}
    assert len(json.dumps(line)) < 1000


def test_the_run_reports_every_leg_it_names():
    src = open(bench.__file__).read()
    body = src[src.index("    line = {\n        \"metric\": METRIC, \"value\": value"):]
    for k in bench.LEGS:
        assert '"%s":' % k in body, k
