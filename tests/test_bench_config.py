"""Both arms of the benchmark state the same configuration (the reference arm runs here, on the CPU)."""
import json
import os
import subprocess
import sys

from conftest import ROOT


def test_reference_arm_states_the_parallelism():
    res = subprocess.run([sys.executable, os.path.join(ROOT, "bench.py"), "--impl", "reference", "--rows", "8",
                          "--cols", "8", "--steps", "1", "--warmup", "0"],
                         check=True, capture_output=True, text=True, cwd=ROOT)
    line = json.loads(res.stdout.strip().split("\n")[-1])
    assert line["impl"] == "reference"
    assert line["config"]["parallelism"] == "1 GPU"
