"""Every index the triangle kernels form (state rows, angle rows, blocks with the padding one) lies inside
what it indexes, for every degree, and the block order is the layout's."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_index_of_every_degree(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "check")
    subprocess.run([nvcc, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2409_19156_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "tri_index_check.cu"), "-o", exe], check=True, capture_output=True)
    done = subprocess.run([exe], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
