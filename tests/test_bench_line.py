"""The benchmark's line stays short enough to be read back whole, however much the
other workloads' legs hold, and loses none of its own figures to them."""

import json

import bench


def test_legs_stay_out_of_the_line():
    own = {k: {"x": 1.0} if k in ("config", "roofline", "e2e", "clocks") else 1.0 for k in bench.LINE_KEYS}
    own["cpu_baseline"] = {"value": 0.05, "kernels": {"sap": "k" * 5000}}
    legs = {f"leg{i}": "v" * 5000 for i in range(4)}
    line, rest = bench.split_line({**legs, **own})
    assert set(line) == set(bench.LINE_KEYS) and set(rest) == set(legs) | {"cpu_baseline_kernels"}
    assert line["cpu_baseline"] == {"value": 0.05} and "kernels" in own["cpu_baseline"]
    assert len(json.dumps(line)) < 2000
