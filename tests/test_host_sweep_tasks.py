"""The sweeps' task lists on the CPU: a C++ harness built from the library's host sources checks
them for one cloth and for batches on either side of every line of the dispatch (96, 192 and
1024 small fronts in a depth; 8 and 40 fronts per SM)."""
import os
import shutil
import subprocess
import tempfile

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2106_05306_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"


def test_tasks():
    cxx = shutil.which("g++")
    if cxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs g++ and the CUDA headers")
    srcs = [os.path.join(ROOT, "tests", "host", "task_check.cpp")] + [
        os.path.join(CSRC, f) for f in ("dc_setup.cpp", "dc_frontal_setup.cpp")]
    # copies and grid size
    cases = [(1, 2), (1, 3), (1, 16), (1, 61), (1, 100), (12, 16), (13, 16), (24, 16), (25, 16), (71, 16), (72, 16),
             (128, 16), (129, 16), (16, 24), (11, 40), (12, 40), (57, 40), (58, 40), (30, 56), (31, 56)]
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "task_check")
        subprocess.check_call([cxx, "-std=c++17", "-O1", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                               "-I", CUDA_INC, *srcs, "-o", exe])
        out = subprocess.run([exe] + [str(v) for c in cases for v in c], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.startswith("ok"), out.stdout + out.stderr
