"""The sines and cosines of the rotary tables (tests/cuda/sincos_check.cu, built with nvcc for sm_103a and run
on the GPU): as accurate as those that the host library gave."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2609_04971_gb300", "csrc")


def test_sines_and_cosines_are_within_half_an_ulp(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "sincos_check")
    subprocess.check_call([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-I", CSRC, "-o",
                           exe, os.path.join(HERE, "cuda", "sincos_check.cu")])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(out.stdout)
    assert out.returncode == 0, out.stdout + out.stderr
