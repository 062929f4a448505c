"""A record that names a neighbour outside the grid raises the request's error
flag in launches of few particles too: a small CUDA program
(tests/cuda/cell_range_check.cu) linked against libmp.so."""
import os
import shutil
import subprocess
import tempfile

import pytest

from paper_2302_13590_gb300 import _build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _program(d):
    exe = os.path.join(d, "cell_range_check")
    lib = _build.build_lib()
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.check_call([nvcc, "-O2", "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-cudart", "shared",
                           "-I", os.path.join(ROOT, "include"), "-I", _build.CSRC,
                           os.path.join(ROOT, "tests", "cuda", "cell_range_check.cu"), lib, "-o", exe,
                           "-Xlinker", "-rpath," + os.path.dirname(lib)])
    return exe


def test_cell_range_check_builds():
    """The check program cross-compiles for sm_103a (no GPU needed)."""
    with tempfile.TemporaryDirectory() as d:
        assert os.path.exists(_program(d))


@pytest.mark.gpu
def test_neighbour_outside_the_grid_is_an_error():
    with tempfile.TemporaryDirectory() as d:
        r = subprocess.run([_program(d)], capture_output=True, text=True, timeout=120)
        print(r.stdout.strip())
        assert r.returncode == 0, r.stdout + r.stderr
