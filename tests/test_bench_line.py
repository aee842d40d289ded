"""The benchmark's line on stdout (no GPU): one line of JSON short enough for a
reader that keeps the last 3,000 characters, the contract's keys whole and
first, whatever the record holds beside them."""
import json
import os
import sys

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


def _record():
    roof = {"kernel": "k" * 60, "bound": "alu", "achieved": 0.123456789012345, "peak": 1.06, "unit": "TFLOP/s",
            "frac": 0.123456789012345, "flops_model": "words " * 60, "traffic": None,
            "runs": [0.1234567890123] * 20}
    sub = {"workload": "w" * 200, "metric": "DOF-iters/s", "value": 1234567890.123456789, "roofline": dict(roof),
           "time_to_tol_ms_mixed": 12.3456789012345, "table": [{"step": i, "iters": i} for i in range(30)],
           "clocks": {"sm_mhz": 2070.0}}
    return {"metric": "m" * 90, "value": 123456789.123456789, "unit": "DOF-iters/s", "n_gpus": 1, "steps": 20,
            "warmup": 5, "ms_per_step": 10.123456789012345, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "w" * 120, "n_dofs": 98127, "timed": "t" * 160, "l2": "flushed"},
            "iters_mixed": 186, "time_to_tol_ms_mixed": 10.123456789012345, "setup_s": 1.23456789,
            "e2e": {"value": 1.23456789012345e9, "unit": "DOF-iters/s", "h2d_bytes_per_step": 785016,
                    "d2h_bytes_per_step": 785016},
            "roofline": roof, "gpu_launches": 12345, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": []},
            "cpu_baseline": {"value": 6.6e6, "unit": "DOF-iters/s", "cores": 1, "kind": "oracle", "sample": "s" * 200},
            "workloads": {f"w{i}": dict(sub) for i in range(8)},
            "rooflines": {f"r{i}": dict(roof) for i in range(6)}, "tiles": {"list": list(range(400))}}


def test_line_is_short_and_keeps_the_contract():
    rec = _record()
    line = bench.short_line(rec)
    assert "\n" not in line and len(line) <= bench.LINE_LIMIT <= 2800
    out = json.loads(line)
    for k in bench.CONTRACT:
        if k in rec:
            assert out[k] == rec[k], k
    assert abs(out["roofline"]["frac"] - rec["roofline"]["frac"]) < 1e-6
    assert out["workloads"]["w3"]["value"] == 1234570000.0
    assert out["iters_mixed"] == 186


def test_short_record_is_kept_whole():
    rec = {k: v for k, v in _record().items() if k in bench.CONTRACT or k in ("iters_mixed",)}
    assert json.loads(bench.short_line(rec)) == rec


def test_record_file(tmp_path, capsys):
    path = tmp_path / "record.json"
    bench.emit(_record(), str(path))
    assert json.loads(path.read_text()) == _record()
    printed = capsys.readouterr()
    assert printed.err == "" and len(printed.out.strip().splitlines()) == 1
