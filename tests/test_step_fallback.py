"""A refused cooperative launch (a process that may use fewer SMs than the device reports): the
default policy streams the rest of the call, GA_RESIDENT_ON reports it.  Host code over stand-ins
for the launchers; no GPU."""
import os
import subprocess

from conftest import ROOT


def test_refused_resident_launch_streams(tmp_path):
    exe = str(tmp_path / "step_fallback_check")
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    csrc = os.path.join(ROOT, "paper_2405_03605_gb300", "csrc")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-I", csrc,
                    "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "cuda", "step_fallback_check.cu"),
                    os.path.join(csrc, "ga_api.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")
    rows = [[int(x) for x in line.split()] for line in out if line]
    # return code, generations launched, generation, resident launches tried, streamed launches
    assert rows[0] == [0, 5000, 5000, 1, 5000]
    assert rows[1] == [0, 5000, 5000, 2, 904]  # the first chunk of 4,096 was resident
    assert rows[2] == [-3, 0, 0, 1, 0]
