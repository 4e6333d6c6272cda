"""The mixed form's direction draw without FP64 (iso_attempt_f32, compiled
for the host): accepts where the FP64 test accepts and returns the FP64
values rounded to FP32, for random draws, draws at the unit circle, near the
origin and at the ends of the range; random draws are almost never left to
FP64, and every draw that is not clear is."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)


def test_integer_attempt_equals_the_fp64_formula(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "direction_probe")
    subprocess.check_call([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"),
                           "-I", os.path.join(ROOT, "paper_1101_4127_gb300", "csrc"),
                           "-o", exe, os.path.join(HERE, "direction_probe.cu")])
    rows = [tuple(map(int, l.split())) for l in subprocess.check_output([exe], text=True).split("\n") if l]
    assert [r[0] for r in rows] == [0, 1, 2, 3]
    assert all(wrong == 0 for _, _, _, wrong in rows), rows
    assert rows[0][2] <= 20, rows          # 4e6 random draws: about 0.4 expected to stay open
