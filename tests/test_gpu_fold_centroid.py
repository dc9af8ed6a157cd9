"""The batched update's fold (tests/cuda/fold_centroid_check.cu, built with nvcc for sm_103a and run on the
GPU) against the functions that it stands for in the common case, bit for bit, and the cases it leaves to them."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_04971_gb300", "csrc")


def test_fold_and_centroid_equals_its_parts(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "fold_centroid_check")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC, "-o",
                           exe, os.path.join(HERE, "cuda", "fold_centroid_check.cu")])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(out.stdout)
    assert out.returncode == 0, out.stdout + out.stderr
