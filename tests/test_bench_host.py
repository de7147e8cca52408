"""bench.py on the CPU: the reference arm (the oracle on the host cores)
prints one JSON line with the contract's keys."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_line_has_the_contract_keys():
    cmd = [sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "2", "--warmup", "1",
           "--grid", "128x64"]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    for k in ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better",
              "scaling", "vs_baseline", "dtype", "data", "config", "impl", "cpu_baseline", "e2e"):
        assert k in d, k
    assert d["impl"] == "reference" and d["unit"] == "MLUPS" and d["higher_is_better"] is True
    assert d["steps"] == 2 and d["warmup"] == 1 and d["value"] > 0
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["cores"] >= 1
    assert d["e2e"]["h2d_bytes_per_step"] == 0 and d["e2e"]["d2h_bytes_per_step"] == 0
    assert "128x64" in json.dumps(d["config"])


def test_roofline_names_the_kernels_that_ran():
    import bench

    label, launches, _ = bench._step_form(["k_phase_l", "k_phase_u", "k_phase_c"])
    assert label.startswith("k_phase_l + k_phase_u + k_phase_c") and launches == 3
    assert bench._step_form(["k_tile"])[1:] == (1, 72) and bench._step_form(["k_step_warp"])[1:] == (1, 72)
    assert bench._step_form(["k_density", "k_update"])[0].startswith("k_update")
    assert bench._step_form(["k_density", "k_update"])[1:] == (2, 88)
    assert bench._ncu_traffic(["k_tile"]) is None  # the committed counters are k_step_warp's
