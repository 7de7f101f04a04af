"""The run that the benchmark's DRAM traffic is captured from does the timed
region's work: one step of each of its lattices in turn."""
import json
import os
import subprocess
import sys

import pytest

import bench

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

pytestmark = pytest.mark.gpu


def test_profile_run_steps_the_timed_lattices_in_turn():
    r = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--profile", "--warmup", "4",
                        "--steps", "10"], capture_output=True, text=True, timeout=300, cwd=ROOT)
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    assert out["lattices"] == bench.LATTICES
    n = 4 + 10
    assert out["steps_of_each"] == [(n - j + bench.LATTICES - 1) // bench.LATTICES
                                    for j in range(bench.LATTICES)]
    assert out["status"] == ["ok"] * bench.LATTICES
