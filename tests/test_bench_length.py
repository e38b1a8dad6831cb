"""The line of the default run is short enough for a reader that keeps a few kilobytes of the output, and --details holds the rest."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
def test_default_line(tmp_path):
    details = tmp_path / "details.json"
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--steps", "3", "--warmup", "3", "--no-cpu-baseline",
                        "--details", str(details)], capture_output=True, text=True, cwd=ROOT, timeout=900)
    assert r.returncode == 0, r.stderr[-2000:]
    (text,) = [x for x in r.stdout.splitlines() if x.startswith("{")]
    assert len(text) <= 6144
    line, full = json.loads(text), json.loads(details.read_text())
    assert set(line) == set(full) and set(line["legs"]) == set(full["legs"]) and len(line["legs"]) == 2
    for key in ("metric", "value", "unit", "ms_per_step", "config", "clocks", "e2e", "gpu_launches"):
        assert line[key] == full[key], key
    for name, leg in line["legs"].items():
        whole = full["legs"][name]
        assert abs(leg["value"] - whole["value"]) <= 1e-4 * whole["value"] and leg["async_wait_timeouts"] == 0
        assert set(whole["roofline"]["per_kernel"]) == set(whole["kernels"])
    assert set(line["roofline"]["per_kernel"]) == set(full["kernels"]) == set(line["kernels"])
