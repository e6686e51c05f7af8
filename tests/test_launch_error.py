"""A launch that fails reports its error and leaves none pending for later calls.  Stand-ins for the
runtime's calls; no GPU."""
import os
import subprocess

from conftest import ROOT


def test_failed_launch_leaves_no_error_pending(tmp_path):
    exe = str(tmp_path / "launch_error_check")
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17",
                    "-I", os.path.join(ROOT, "paper_2405_03605_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "cuda", "launch_error_check.cu"), "-o", exe], check=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True).stdout
    assert out.split() == ["1", "0"] * 3
