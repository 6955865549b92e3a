"""The line the benchmark prints: short enough to be read back whole, with every
key of the contract, whatever the sections hold."""

import json

import bench

CONTRACT = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "clocks", "e2e", "gpu_launches", "cpu_baseline", "roofline")


def test_line_is_short_and_whole():
    table = {f"{f}B/{c}": 0.123456789012345 for f in (32, 64, 128) for c in range(40)}
    num = 87654321.12345678
    out = {k: num for k in CONTRACT}
    out.update(metric=bench.METRIC, unit=bench.UNIT, scaling="weak", vs_baseline=None, dtype="c64", data="synthetic",
               config=dict(bench.workload_config(8192), qubit_layout={"rows": list(range(14))}, schedule=table),
               roofline=dict({k: num for k in bench.LINE_KEYS["roofline"]}, touch_floor_note="x" * 300),
               clocks={"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": ["sw_power_cap"]},
               e2e=dict(value=num, unit=bench.UNIT, h2d_bytes_per_step=num, d2h_bytes_per_step=num,
                        api="tq_evolve_taylor5_batch_support_host (states in pinned host memory)", tune=table),
               cpu_baseline={"value": num, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "y" * 200},
               serving={"sweep": [table] * 50}, spmv=table)
    line = bench.headline_line(out)
    got = json.loads(line)
    assert "\n" not in line and len(line) < 3000
    assert all(k in got for k in CONTRACT)
    assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(got["e2e"])
    assert got["clocks"] == out["clocks"] and got["value"] == num and got["config"]["n_states"] == 8192
    assert "serving" not in got and "schedule" not in got["config"]
