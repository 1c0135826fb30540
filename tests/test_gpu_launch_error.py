"""A refused launch of a step kernel leaves no error behind for the next call: compiles
tests/launch_error_check.cu (the library's own launch header) with nvcc and runs it."""
import os
import shutil
import subprocess

import pytest

from paper_2301_01622_gb300 import build as B

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_refused_launch_is_reported_once(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "launch_error_check")
    src = os.path.join(ROOT, "tests", "launch_error_check.cu")
    r = subprocess.run([nvcc, *B.ARCH, "-std=c++17", "-I", B.CSRC, src, "-o", exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "launch error check ok" in r.stdout, r.stdout[-2000:]
