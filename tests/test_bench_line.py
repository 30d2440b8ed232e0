"""The line that bench.py prints holds the contract's keys and stays short however much the full
record holds. No GPU."""
import importlib.util
import json
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_the_line_is_short_and_complete():
    spec = importlib.util.spec_from_file_location("bench_line_under_test", os.path.join(ROOT, "bench.py"))
    b = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(b)
    record = {k: 1.0 / 3.0 for k in b.CONTRACT_KEYS}
    record.update(mixed_vs_fp64_at_equal_l2={"direct": {"mixed_l2_vs_exact": 4e-7, "fp64_l2_vs_exact": 4e-7}},
                  center_stencils={"mixed": {"value": 3e7, "more": ["x"] * 1000}}, served={"requests": ["y" * 100] * 500},
                  cpu_baseline={"value": 4e4, "unit": "u", "cores": 16, "kind": "oracle", "sample": "z" * 5000})
    line = b.contract_line(record)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "roofline"):
        assert k in line
    assert len(json.dumps(line)) < 2000
    record["cpu_baseline"] = None
    assert b.contract_line(record)["cpu_baseline"] is None
