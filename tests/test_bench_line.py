"""The benchmark's printed line holds the launch contract's keys and stays short enough to be
read from the end of a run's output, however long the legs' own records are."""

import importlib.util
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
X = 0.12345678901234567


def load():
    spec = importlib.util.spec_from_file_location("bench", os.path.join(ROOT, "bench.py"))
    m = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(m)
    return m


def record(bench):
    """A full record with every leg, the numbers at full length and a long series in each leg."""
    full = {k: X for k in bench.CONTRACT}
    full["metric"] = bench.METRIC
    full["config"] = {f"option_{i}": "a setting of the workload" for i in range(11)}
    for block, paths in bench.KEPT.items():
        full[block] = {"series": [{"w": i, "q": X} for i in range(286)]}
        for path in paths:
            d = full[block]
            *way, last = path.split(".")
            for k in way:
                d = d.setdefault(k, {})
            d[last] = X
    full["cpu_baseline"]["sample"] = "the first 2 buffers (2^22 samples each) of the same stream, single thread"
    return full


def test_line_is_short_and_complete():
    bench = load()
    full = record(bench)
    line = bench.short_line(full)
    assert len(json.dumps(full)) > 100_000 and len(json.dumps(line)) <= bench.LINE_MAX
    for k in bench.CONTRACT:
        assert line[k] == full[k]
    contract = {"e2e": ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"),
                "clocks": ("sm_mhz", "sm_max_mhz", "reasons"), "cpu_baseline": ("value", "cores", "kind", "sample")}
    for block, keys in contract.items():
        for k in keys:
            assert line[block][k] == full[block][k]
    assert set(line) == set(bench.CONTRACT) | set(bench.KEPT)


def test_legs_that_did_not_run_are_left_out():
    bench = load()
    full = record(bench)
    full["cnn"] = full["stability"] = None
    line = bench.short_line(full)
    assert "cnn" not in line and "stability" not in line and "batched" in line


def test_only_the_short_line_is_printed():
    src = open(os.path.join(ROOT, "bench.py")).read()
    arm = src[src.index("def gpu_arm"):]
    arm = arm[:arm.index("\ndef ")]
    prints = [l.strip() for l in arm.splitlines() if l.strip().startswith("print(") and "stderr" not in l]
    assert prints == ["print(json.dumps(short_line(line)), flush=True)"]
