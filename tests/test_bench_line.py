"""The benchmark's report is one line and stays short: a timing record does not grow
with the number of timed calls."""
import importlib.util
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_a_timing_record_does_not_grow_with_its_calls():
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    bench = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(bench)
    clocks = {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 4}
    short, long = (bench.timing_record([1.0 + i / 7.0 for i in range(k)], clocks) for k in (4, 400))
    assert long["reps"] == 400 and long["min_ms"] == 1.0 and long["max_ms"] == 1.0 + 399 / 7.0
    assert len(json.dumps(long)) <= len(json.dumps(short)) + 100
