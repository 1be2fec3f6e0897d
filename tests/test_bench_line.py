"""The benchmark's output line: one JSON object with the headline's keys, short enough that a
log's last 1,500 characters hold it whole, and everything measured in the legs file."""
import argparse
import json

import bench


def test_line_is_short_and_legs_are_kept(tmp_path, capsys):
    args = argparse.Namespace(chains=256, iters_per_step=1000)
    line = {"metric": bench.METRIC, "value": 341234567.8901234, "unit": bench.UNIT, "n_gpus": 1, "steps": 200, "warmup": 10,
            "ms_per_step": 0.7512345678901234, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic", "config": bench.run_config(args),
            "e2e": {"value": 339876543.2109876, "unit": bench.UNIT, "h2d_bytes_per_step": 60060,
                    "d2h_bytes_per_step": 32468, "note": "n" * 300},
            "gpu_launches": 123456,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "power_w": 812.5, "samples": 1234,
                       "reasons": ["sw_power_cap"]},
            "roofline": {"kernel": "k", "bound": "alu", "unit": "warp instructions/s", "achieved": 9.87654321012345e11,
                         "peak": 1.2345678901234e12, "frac": 0.8012345678901234, "traffic": 1.9e6, "note": "x" * 2000},
            "cpu_baseline": {"value": 23.07289265, "unit": bench.UNIT, "cores": 16, "kind": "oracle", "sample": "s" * 500},
            "score_orders": {"by_orders": [{"orders": i, "ms": 0.1} for i in range(200)]}}
    path = tmp_path / "legs.json"
    bench.emit(line, str(path))
    out = capsys.readouterr().out
    assert out.count("\n") == 1 and len(out) <= 1500, len(out)
    head = json.loads(out)
    for k in bench.HEAD_KEYS:
        assert head[k] == (line[k] if k != "e2e" else {x: y for x, y in line["e2e"].items() if x != "note"}), k
    assert json.loads(path.read_text()) == line
    # a place that cannot be written costs the file, not the line
    bench.emit(line, str(tmp_path / "none" / "legs.json"))
    assert json.loads(capsys.readouterr().out)["value"] == line["value"]
