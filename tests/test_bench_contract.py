"""The JSON line of bench.py's reference arm (the CPU oracle timed on the host cores) carries the keys the
measurement contract names.  Runs the smallest workload; no GPU."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_one_contract_line():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--workload", "cfg1",
                          "--steps", "1", "--warmup", "0"], capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert out.returncode == 0, out.stderr[-2000:]
    lines = [l for l in out.stdout.splitlines() if l.strip()]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference"
    for key in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
                "vs_baseline", "dtype", "data", "config", "cpu_baseline", "e2e"):
        assert key in d, key
    assert d["metric"] == "expanded_layer_tokens_per_s" and d["unit"] == "tokens/s" and d["value"] > 0
    assert d["config"]["workload"] == "cfg1"
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1 and d["cpu_baseline"]["sample"]
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0
    assert d["e2e"]["value"] == d["value"]


def test_the_line_keeps_its_numbers_to_six_digits():
    import bench
    got = bench.short({"a": 1.23456789, "b": [2, 3.0000001, None], "c": {"d": 6085240.885966282, "e": "x", "f": True}})
    assert got == {"a": 1.23457, "b": [2, 3.0, None], "c": {"d": 6085240.0, "e": "x", "f": True}}
