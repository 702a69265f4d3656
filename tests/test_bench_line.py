"""The benchmark's one line of output stays short enough to be kept whole by what collects it
(some keep the last 8,000 characters of a program's output): the legs' tables go to stderr."""
import json
import os
import sys

sys.path.insert(0, os.path.join(os.path.dirname(__file__), ".."))
import bench  # noqa: E402


def test_line_is_short():
    prof = {f"kernel_name_{i:02d}": (60, 123.45678901234567) for i in range(14)}
    leg = dict(value=12345.678901234567, ms_per_step=123.45678901234567, schedule=dict(a=1, b=16, c=0, d=2), kernels=bench.kernel_table(prof),
               err_vs_fp64={k: 1.2345678901234567e-14 for k in ("K", "R", "du", "dq")}, precision="x" * 150,
               roofline={f"entry_{i}": 0.12345678901234567 for i in range(12)}, gpu_launches=320)
    line = {"metric": "m" * 80, "kernels": bench.kernel_table(prof), "config": {"workload": "w" * 300}, "roofline": leg["roofline"],
            "cpu_baseline": "c" * 400, "mixed": dict(leg), "mixed_orders": {"workload": "w" * 100, "fp64": dict(leg), "mixed": dict(leg)},
            "extras": {f"measurement_{i}": {"ms": 1.2345678901234567, "text": "t" * 100} for i in range(6)}}
    low = {f"low_precision_leg_{i}": dict(leg) for i in range(5)}
    out = bench.short(bench.slim(line, low))
    assert len(json.dumps(out)) < 8000
    assert out["mixed"]["kernels"]["kernel_name_03"] == 123.5 and out["low_precision_leg_2"]["err_vs_fp64"]["du"] > 0
    assert line["mixed"]["kernels"]["kernel_name_03"]["launches"] == 60             # the full tables are untouched
