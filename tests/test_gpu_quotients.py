"""The step kernels' quotients by a reciprocal and a correction give the bits of
correctly rounded divisions (tests/native/quotient_check.cu: 16.8 M of each)."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

pytestmark = pytest.mark.gpu


def test_quotients_are_the_divisions(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "quotient_check")
    subprocess.check_call([nvcc, "-std=c++17", "-O3", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_2012_14707_gb300", "csrc"),
                           "-o", exe, os.path.join(HERE, "native", "quotient_check.cu")])
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0, out.stdout + out.stderr
