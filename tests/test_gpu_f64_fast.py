"""The FP64 step's short forms (log1p with its row from FP32, the motion
without a branch, FP32 truncation and time keys on the words of a double, the
screened exit axis) against the general forms, bit for bit: a small CUDA
program (tests/cuda/f64_fast_check.cu) built for sm_103a and run on the GPU."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
def test_short_forms_match_general_forms():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "f64_fast_check")
        subprocess.check_call([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-fmad=false",
                               "-I", os.path.join(ROOT, "include"),
                               "-I", os.path.join(ROOT, "paper_2302_13590_gb300", "csrc"),
                               os.path.join(ROOT, "tests", "cuda", "f64_fast_check.cu"), "-o", exe])
        r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
        print(r.stdout.strip())
        assert r.returncode == 0, r.stdout + r.stderr
