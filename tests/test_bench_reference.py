"""The reference arm of bench.py (the CPU oracle on the host cores) runs without a GPU: its JSON line is checked
here at a shrunk size; the default size is the same code path with 128 tables."""
import json
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_reference_arm_prints_the_contract_line():
    out = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--steps", "2",
                          "--warmup", "3", "--requests", "2", "--layers", "1"],
                         cwd=ROOT, capture_output=True, text=True, timeout=600, check=True).stdout
    lines = [l for l in out.splitlines() if l.startswith("{")]
    assert len(lines) == 1
    d = json.loads(lines[0])
    assert d["impl"] == "reference" and d["unit"] == "GB/s" and d["higher_is_better"] is True
    assert d["n_gpus"] == 1 and d["steps"] == 2 and d["warmup"] == 3 and d["scaling"] == "weak"
    assert d["vs_baseline"] is None and d["data"] == "synthetic" and "workload" in d["config"]
    assert d["value"] > 0 and d["ms_per_step"] > 0
    assert d["cpu_baseline"]["kind"] == "oracle" and d["cpu_baseline"]["value"] == d["value"]
    assert d["cpu_baseline"]["cores"] >= 1 and d["cpu_baseline"]["sample"]
    assert d["e2e"] == {"value": d["value"], "unit": "GB/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}
    assert 0.5 < d["hit_rate"] < 1.0


def test_other_ranks_of_the_reference_arm_do_nothing():
    env = dict(os.environ, RANK="1", WORLD_SIZE="2", LOCAL_RANK="1")
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--gpus", "2",
                        "--steps", "1", "--warmup", "3"], cwd=ROOT, env=env, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip() == ""


def test_clocks_where_the_first_sample_comes_late(tmp_path, monkeypatch):
    """A very short run on a busy host: it is over before nvidia-smi has written its first line."""
    tool = tmp_path / "nvidia-smi"
    tool.write_text('#!/bin/sh\nsleep 0.6\nwhile true; do echo "1900, 1965, 200, Not Active, Not Active, Not Active, Active"; sleep 0.1; done\n')
    tool.chmod(0o755)
    monkeypatch.setenv("PATH", str(tmp_path) + os.pathsep + os.environ["PATH"])
    monkeypatch.syspath_prepend(ROOT)
    import bench
    sampler = bench.ClockSampler(0)
    sampler.start()
    got = sampler.stop()
    assert got["sm_mhz"] == 1900 and got["sm_max_mhz"] == 1965 and got["reasons"] == ["sw_power_cap"]
