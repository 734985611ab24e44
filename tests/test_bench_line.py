"""The benchmark's printed line holds its contract's fields and fits into the last
3000 bytes of the output, however many rows lie behind it; the rows go to stderr."""
import json

import bench


def _out():
    kernel = {"kernel": "k" * 30, "timed": "t" * 60, "bytes_per_unit": "b" * 200, "duration_ms": 0.8139278173446655,
              "algorithmic_bytes": 360771212.5576341, "achieved_gbs": 402.86946059743485, "traffic": None}
    sweep = {f"{t:g}": {f"field_{i}": 0.123456789012345 for i in range(12)} for t in (0.0, 0.01, 0.05, 0.1)}
    cfg = {"workload": "w" * 200, "paths": 3_000_000, "max_bounces": 7, "mode": "error", "tau": 0.01, "frames_timed": 20,
           "l2": "inputs larger than L2 (path buffers 816 MB)", "reuse_ms_per_frame": 1.0904512405395508,
           "trace_all_ms_per_frame": 3.7221584320068, "speedup_vs_trace_all": 3.41341345, "rays_per_frame_reuse": 1343434.05,
           "rays_per_frame_trace_all": 9343434.9, "listed_per_frame": 391493.35, "device_status": [0, 0],
           "kernels": [kernel] * 7, "tau_sweep": sweep, "modes_tau_1pct": sweep,
           "city": {"reuse_ms_per_frame": 0.4012345, "kernels": [kernel] * 7}, "batch16": {"batch_frame_ms": 0.9876, "x": sweep}}
    return {"metric": bench.METRIC, "value": 2751169742.5, "unit": "paths/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 1.0904512405395508, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic", "config": cfg,
            "roofline": {"kernel": "k" * 100, "bound": "alu", "achieved": 2.6289709588, "peak": 38.6134, "unit": "Top/s",
                         "frac": 0.0680815, "traffic": None, "traffic_note": "n" * 80, "duration_ms": 0.8955,
                         "peak_kind": "p" * 90, "algorithmic_ops": 2354254003.75, "ops_rule": "o" * 150,
                         "hbm": {"achieved": 402.8, "peak": 6677.2, "unit": "GB/s", "frac": 0.06, "peak_kind": "measured"},
                         "kernels": [kernel] * 7, "source_digest": "0123456789abcdef"},
            "gpu_launches": 80, "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 55},
            "e2e": {"value": 2441169742.5, "unit": "paths/s", "h2d_bytes_per_step": 1024, "d2h_bytes_per_step": 12582912},
            "cpu_baseline": {"value": 488.9, "unit": "paths/s", "cores": 16, "kind": "oracle", "sample": "s" * 250,
                             "frame_s": {"2": 0.4, "15": 0.4, "30": 0.4}, "ambiguity": {"x": 1, "y": 2}}}


def test_line_is_short_and_whole(capsys):
    out = _out()
    bench.emit(out)
    got = capsys.readouterr()
    lines = got.out.splitlines()
    assert len(lines) == 1 and len(lines[0]) <= bench.LINE_BYTES < 3000
    d = json.loads(lines[0])
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
              "vs_baseline", "dtype", "data", "gpu_launches", "e2e", "clocks"):
        assert d[k] == out[k], k
    assert d["config"]["workload"].startswith("w" * 100)
    assert abs(d["config"]["city_reuse_ms_per_frame"] - 0.4012345) < 1e-6
    assert d["roofline"]["frac"] == 0.0680815
    assert json.loads(got.err)["details"] == json.loads(json.dumps(out))
