"""`bench.py --impl reference` runs as many epochs as it is asked for (the handles of the pool's blocks
have to last for all of them) and prints its line."""
import json
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("config", [1, 5])
def test_reference_arm(config):
    r = subprocess.run([sys.executable, "bench.py", "--impl", "reference", "--config", str(config), "--scale", "0.004",
                        "--steps", "20", "--warmup", "5"], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, CUDA_VISIBLE_DEVICES=""))
    assert r.returncode == 0, r.stderr[-2000:]
    line = json.loads(r.stdout.strip().splitlines()[-1])
    assert line["impl"] == "reference" and line["steps"] == 20 and line["warmup"] == 5
    assert line["value"] > 0 and line["config"]["pool"] == config
