"""The FP64 quotient and reciprocal of the per-cell update and the FP64 walk,
which replace the division, and the FP32 to FP64 widening, which replaces the
conversion, give the same bits (compiled from the kernels' own header)."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_quotient_reciprocal_and_widening_are_exact(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "division_probe")
    subprocess.check_call([nvcc, "-std=c++17", "-O2", "-gencode", "arch=compute_103a,code=sm_103a",
                           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1101_4127_gb300", "csrc"),
                           "-o", exe, os.path.join(HERE, "division_probe.cu")])
    counts = [int(v) for v in subprocess.check_output([exe], text=True).split()]
    assert counts == [0] * 11
