"""The benchmark's stdout line stays short: the headline record and one value
per other workload, whose full records go to stderr."""
import json

import bench


def test_headline_line_is_short_and_complete():
    rec = {"value": 1.0e7, "unit": "grid-pt-steps/s", "config": {"workload": "x" * 300}, "roofline": {"note": "y" * 2000}}
    out = {"metric": "m", "value": 2.0, "e2e": {"value": 3.0}, "clocks": {"sm_mhz": 2070}, "gpu_launches": 5,
           "config": {"workload": "z" * 200}, "cpu_baseline": {"value": 1.0}}
    want = dict(out)
    for k in bench.OTHER_WORKLOADS:
        out[k] = dict(rec)
    out["c4"] = {"error": "no room"}
    out["alpha_p8"] = {"alpha": 0.1, "pfasst": [rec] * 5}
    line = bench.headline(out)
    others = line.pop("other_workloads")
    assert line == want
    assert others["mixed"] == 1.0e7 and others["c4"] == "no room" and others["alpha_p8"] == 0.1
    assert set(others) == set(bench.OTHER_WORKLOADS)
    assert len(json.dumps(bench.headline(out))) < 3000
    assert bench.headline(want) == want
