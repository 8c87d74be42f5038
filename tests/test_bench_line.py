"""bench.py's result line stays short whatever the record holds, and keeps every figure the metric is judged by (CPU)."""
import json
import os
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

CONTRACT = {"metric": "merged points/sec", "value": 6178604.549114504, "unit": "points/s", "n_gpus": 1, "steps": 20, "warmup": 5,
            "ms_per_step": 161.84884338378907, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic", "gpu_launches": 595,
            "clocks": {"sm_mhz": 2070.0, "sm_max_mhz": 2070.0, "reasons": [], "samples": 21}}


def _record(steps):
    kernels = {f"k_kernel_{i}": {"launches": 60, "ms": 140.07788701355457 + i} for i in range(35)}
    roof = {"kernel": "k_join", "per_launch_ms": 6.904369879679548, "traffic": None, "bound": "hbm", "unit": "GB/s",
            "peak": 6779.0, "peak_kind": "measured copy (hbm_gbs), of measured", "achieved": 975.8034002729344, "frac": 0.14394}
    sub = {"workload": "w" * 140, "value": 384624.03446667054, "unit": "points/s", "ms_per_step": 2599.94, "form": "f" * 100,
           "kernels": kernels, "merge_stats": {f"s{i}": 2539157793 for i in range(12)}, "roofline_by_kernel": {"a": roof, "b": roof},
           "sizes": list(range(10_000, 10_064)), "plain_fp32": {"value": 1.0, "same_graph": True}, "recall@10": 0.4486}
    times = [161.83421325683594 + 1e-6 * i for i in range(steps)]
    return {**CONTRACT, "config": {"workload": "Sift-like merge " + "x" * 130, "N": 1_000_000, "d": 128},
            "e2e": {"value": 5945277.421674175, "unit": "points/s", "h2d_bytes_per_step": 640000000,
                    "d2h_bytes_per_step": 132000004, "step_wall_ms": times, "step_device_ms": times},
            "roofline": roof, "cpu_baseline": {"value": 18192.1, "unit": "points/s", "cores": 16, "kind": "oracle", "sample": "s" * 150},
            "roofline_by_kernel": {"k_cross_query": roof, "k_join": roof, "k_prune": roof}, "kernels": kernels, "step_ms": times,
            "plain_fp32": {"value": 1940582.4, "ms_per_step": 515.3, "same_graph": True, "form": "f" * 50},
            "configs": {**{n: sub for n in ("small", "precision", "fp8", "batched")}, "bad": {"error": "RuntimeError: " + "e" * 5000}}}


def test_line_is_short_and_keeps_the_contract():
    import bench
    for steps in (5, 200):
        rec = _record(steps)
        text = json.dumps(bench.headline(rec))
        assert len(text) < 4096, len(text)
        line = json.loads(text)
        for k, v in CONTRACT.items():
            assert line[k] == v or abs(line[k] / v - 1) < 1e-6, k
        assert line["config"]["N"] == 1_000_000
        assert {"value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step"} <= set(line["e2e"])
        assert line["roofline"]["kernel"] == "k_join" and line["plain_fp32"]["same_graph"] is True
        assert set(line["configs"]) == set(rec["configs"]) and line["configs"]["fp8"]["value"] > 0


def test_headline_leaves_the_record_alone():
    import bench
    rec = _record(5)
    before = json.dumps(rec)
    bench.headline(rec)
    assert json.dumps(rec) == before
