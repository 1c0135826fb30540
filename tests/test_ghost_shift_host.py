"""Host check of the distance to a node's ghost copy: compiles
tests/ghost_shift_check.cu (the library's own layout header, host code only) with nvcc
and runs it."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_ghost_distances_of_long_rows(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "ghost_shift_check")
    src = os.path.join(ROOT, "tests", "ghost_shift_check.cu")
    inc = os.path.join(ROOT, "paper_2301_01622_gb300", "csrc")
    r = subprocess.run([nvcc, "-std=c++17", "-I", inc, src, "-o", exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "ghost shift check ok" in r.stdout, r.stdout[-2000:]
