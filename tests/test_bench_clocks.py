"""bench.py's clock record covers the timed region, however long nvidia-smi takes to start (a stand-in for it, no GPU)."""
import os
import sys
import time

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

SLOW_START = """#!/bin/sh
sleep 0.7
echo "0, 120, 1965, 100, 0x0, Not Active, Not Active, Not Active, Not Active"
while true; do
    sleep 0.02
    echo "0, 1965, 1965, 300, 0x0, Not Active, Not Active, Not Active, Active"
done
"""


def test_samples_of_a_short_region(monkeypatch, tmp_path):
    import bench
    smi = tmp_path / "nvidia-smi"
    smi.write_text(SLOW_START)
    smi.chmod(0o755)
    monkeypatch.setenv("PATH", f"{tmp_path}:{os.environ['PATH']}")
    sampler = bench.ClockSampler(0)
    time.sleep(0.5)
    clocks = sampler.stop()
    assert clocks["samples"] >= 3                       # twenty or so on an idle machine
    assert clocks["sm_mhz"] == 1965.0 and clocks["reasons"] == ["sw_power_cap"]


def test_no_nvidia_smi(monkeypatch, tmp_path):
    import bench
    monkeypatch.setenv("PATH", str(tmp_path))
    assert bench.ClockSampler(0).stop()["sm_mhz"] is None
