"""The benchmark prints one JSON line with the keys and units the harness reads: the
GPU arm on a small grid (GPU), and the reference arm, which times the oracle on the
host (CPU)."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def run_bench(*args, timeout=600):
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), *args], capture_output=True, text=True,
                       timeout=timeout, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [x for x in r.stdout.strip().splitlines() if x.startswith("{")]
    assert len(lines) == 1, r.stdout[-2000:]
    return json.loads(lines[0])


COMMON = {"metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
          "vs_baseline", "dtype", "data", "config"}


def test_reference_arm_line():
    d = run_bench("--impl", "reference", "--steps", "1", "--warmup", "3")
    assert COMMON <= set(d) and d["impl"] == "reference"
    assert d["value"] > 0 and d["unit"] == "amp-updates/s" and d["higher_is_better"] is True
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["cores"] >= 1 and cb["value"] == d["value"] and cb["sample"]
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0
    assert "workload" in d["config"]


@pytest.mark.gpu
def test_gpu_arm_line():
    d = run_bench("--rows", "2", "--cols", "7", "--steps", "2", "--warmup", "3")
    assert COMMON <= set(d)
    assert d["n_gpus"] == 1 and d["steps"] == 2 and d["warmup"] == 3 and d["scaling"] == "weak"
    assert d["value"] > 0 and d["dtype"] == "f64" and d["data"] == "synthetic" and "workload" in d["config"]
    rf = d["roofline"]
    assert rf["bound"] == "hbm" and rf["unit"] == "GB/s" and rf["achieved"] > 0 and "traffic" in rf
    if rf["peak"]:
        assert rf["frac"] == pytest.approx(rf["achieved"] / rf["peak"])
    e = d["e2e"]
    assert e["value"] > 0 and e["unit"] == d["unit"] and e["h2d_bytes_per_step"] > 0 and e["d2h_bytes_per_step"] > 0
    assert d["gpu_launches"] > 0
    assert {"sm_mhz", "sm_max_mhz", "reasons"} <= set(d["clocks"])
    cb = d["cpu_baseline"]
    assert cb["kind"] == "oracle" and cb["value"] > 0 and cb["cores"] >= 1
    assert 0.0 < d["fidelity"] <= 1.0 + 1e-12 and d["fidelity"] >= d["fidelity_lb_sum"] - 1e-12


@pytest.mark.gpu
def test_value_times_the_call_that_a_user_makes():
    """The timed steps run as the end-to-end steps do, by groups of gates (a gate by itself
    takes three launches); the gates timed one by one are reported beside them."""
    d = run_bench("--rows", "4", "--cols", "5", "--steps", "3", "--warmup", "3", "--no-cpu-baseline", "--no-sweep",
                  "--no-batch")
    assert 0 < d["gpu_launches"] < 2 * d["config"]["gates_timed"]
    g = d["gate_by_gate"]
    assert g["gates"] == sum(c["launches"] for c in d["roofline_by_class"].values()) > 0
    assert d["value"] > 0 and g["amp_updates_per_s"] > 0
