"""The benchmark's result line is short enough to be kept whole: its long tables go to standard error."""
import json


def test_long_tables_leave_the_line():
    import bench
    sweep = {"workload": "w" * 160, "opening_angle": [{"theta": 0.1 * k} for k in range(100)]}
    per = [{"kind": "plummer", "n": 206866, "median": 0.0014251246831051717, "p99": 0.007422632330057729}] * 64
    line = {"metric": bench.METRIC, "value": 1.0, "e2e": {"value": 2.0}, "gpu_launches": 3,
            "error": {"plummer_2p13": {"median": 1e-3}, "sweeps_plummer_2p13": sweep},
            "batch": {"speedup_vs_serial": 2.9, "error_vs_fp64_direct": {"max_p99": 0.01, "per_system": per}}}
    before = json.dumps(line)
    short, tables = bench.split_tables(line)
    assert json.dumps(line) == before  # (not changed in place)
    assert tables == {"sweeps_plummer_2p13": sweep, "batch_errors_per_system": per}
    assert short["error"] == {"plummer_2p13": {"median": 1e-3}}
    assert short["batch"] == {"speedup_vs_serial": 2.9, "error_vs_fp64_direct": {"max_p99": 0.01}}
    assert {k: v for k, v in short.items() if k not in ("error", "batch")} == {
        k: v for k, v in line.items() if k not in ("error", "batch")}
    assert len(json.dumps(short)) < 1000
    for none in ({}, {"error": None, "batch": None}, {"error": {"a": 1}, "batch": {"x": 2}}):
        assert bench.split_tables(none) == (none, {})
