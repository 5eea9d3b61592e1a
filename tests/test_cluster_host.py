"""The largest cluster that decodes a frame, for devices that run fewer blocks together
(host code with a stand-in for the occupancy query; no GPU needed)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_largest_cluster_falls_back_to_smaller_ones_and_to_none(tmp_path):
    nvcc = shutil.which("nvcc") or ("/usr/local/cuda/bin/nvcc" if os.path.exists("/usr/local/cuda/bin/nvcc") else None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "largest_cluster")
    subprocess.check_call([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2508_03567_gb300", "csrc"),
                           os.path.join(HERE, "c", "largest_cluster.cu"), "-o", exe])
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    rows = [tuple(int(x) for x in out[i:i + 3]) for i in range(0, len(out), 3)]
    # blocks the device runs together: largest cluster with, and without, sizes beyond 8
    assert rows == [(16, 16, 8), (8, 8, 8), (4, 4, 4), (2, 2, 2), (1, 0, 0), (0, 0, 0)]
