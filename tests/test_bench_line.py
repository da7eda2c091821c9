"""bench.py's output: one short JSON line on stdout, the full record on stderr."""
import json


def test_headline_is_one_short_line(capsys):
    import bench
    big = {k: "x" * 40 for k in ("a", "b")}
    line = {"metric": "FP64 node-steps/s", "value": 10431520850.732428, "unit": "node-steps/s", "n_gpus": 1, "steps": 100,
            "warmup": 5, "ms_per_step": 9.576488934783265, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic", "config": {"workload": "w" * 120, "l2": "l" * 200, "parallelism": "single"},
            "e2e": {"value": 8837009438.283354, "unit": "node-steps/s", "h2d_bytes_per_step": 1.5, "d2h_bytes_per_step": 2.5,
                    "per_iteration_ms": list(range(1000))},
            "gpu_launches": 1300, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 23},
            "roofline": {"kernel": "node_pass", "bound": "hbm", "achieved": 1.0, "peak": 2.0, "unit": "GB/s", "frac": 0.5,
                         "traffic": 1.0, "share_of_timed_region": 0.4, "peak_note": "n" * 300},
            "cpu_baseline": {"value": 1.0, "unit": "node-steps/s", "cores": 16, "kind": "oracle", "sample": "s" * 160},
            "rings": [big] * 100, "served": big, "peaks": big}
    bench.print_line(line)
    out, err = capsys.readouterr()
    assert out.count("\n") == 1 and len(out) <= bench.HEADLINE_MAX + 1
    got = json.loads(out)
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling", "vs_baseline",
              "dtype", "data", "config", "gpu_launches", "clocks"):
        assert got[k] == line[k]
    assert set(got["e2e"]) == {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"}
    assert json.loads(err.split("bench detail: ", 1)[1]) == line
