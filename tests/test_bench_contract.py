"""The benchmark's reference arm and helpers, on CPU: JSON contract of the printed line."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_one_json_line_with_the_contract_keys():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "1",
                          "--warmup", "0"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert out.returncode == 0, out.stderr
    lines = [ln for ln in out.stdout.splitlines() if ln.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    for key in ("impl", "metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
                "scaling", "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert key in d, key
    assert d["impl"] == "reference" and d["higher_is_better"] is False and d["unit"] == "us"
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] == 1
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["value"] == d["value"] > 0
    assert "workload" in d["config"] and "model" not in d["config"]


def test_reference_arm_is_silent_on_other_ranks():
    env = dict(os.environ, RANK="1", WORLD_SIZE="2", LOCAL_RANK="1")
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--gpus", "2",
                          "--steps", "1", "--warmup", "0"], capture_output=True, text=True, timeout=120, cwd=ROOT, env=env)
    assert out.returncode == 0 and out.stdout.strip() == ""


def test_peak_lookup_and_percentiles():
    sys.path.insert(0, ROOT)
    import bench
    peak, kind = bench.read_peaks()
    assert peak > 1000 and kind in ("measured", "fallback")
    assert bench.pct([1, 2, 3, 4, 5], 50) == 3


def test_the_line_for_stdout_is_short_and_has_the_contract_keys():
    sys.path.insert(0, ROOT)
    import bench
    table = {str(i): {"p50_us": 1.234567, "note": "x" * 80} for i in range(200)}
    record = {
        "metric": bench.METRIC, "value": 0.928, "unit": "us", "n_gpus": 1, "steps": 400, "warmup": 20, "ms_per_step": 0.06543,
        "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "accumulator": "f32",
        "data": "synthetic", "config": {"workload": "w" * 200, "l2": "l" * 200, "replicas": 1}, "p99_us": 0.96,
        "us_per_allreduce_mean": 1.02, "roofline": {"bound": "hbm", "achieved": 6500.0, "peak": 6541.5, "unit": "GB/s",
                                                    "frac": 0.99, "kernel": "k" * 80, "other_modes": table},
        "roofline_decode": table, "cpu_baseline": {"value": 2800.0, "unit": "us", "cores": 1, "kind": "oracle", "sample": table},
        "e2e": {"value": 18.0, "unit": "us", "p99": 19.0, "h2d_bytes_per_step": 4194304, "d2h_bytes_per_step": 524288,
                "what": "y" * 500},
        "by_payload": table, "gpu_launches": 400,
        "clocks": {"sm_mhz": 1965.0, "sm_max_mhz": 1965.0, "reasons": ["sw_power_cap"]},
        "speculation": table, "detail": table, "paper_context": "z" * 300}
    text = json.dumps(bench.headline(record))
    assert len(text) < 3000
    line = json.loads(text)
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "gpu_launches", "clocks", "e2e", "roofline", "cpu_baseline"):
        assert key in line and line[key] == record[key] or isinstance(line[key], dict), key
    assert line["e2e"]["h2d_bytes_per_step"] == 4194304 and line["clocks"] == record["clocks"]
    # sections that were left out (--only) are absent there, too
    assert bench.headline({**record, "e2e": None, "roofline": None, "cpu_baseline": None})["e2e"] is None
