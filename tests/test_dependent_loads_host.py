"""Kernels launched as programmatic dependents live while the kernel before them still
writes what they will read, so none of them reads it with the non-coherent load: no
__ldg, and no const __restrict__ pointer to data that the compiler could turn into one."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2301_01622_gb300", "csrc")


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_dependent_kernels_read_coherently():
    launched = set()
    for name in sorted(os.listdir(CSRC)):
        launched |= set(re.findall(r"launch_overlapped\(\s*(\w+)", _read(name)))
    assert launched - {"void"} <= {"k_moment_pair", "k_cg_pair", "kern"}  # the files below hold all of them
    adjoint = _read("adjoint.cu")
    start = adjoint.index("struct Adjoint {")
    parts = {n: _read(n) for n in ("moment_pair.cuh", "cg_pair.cuh", "pair_march.cuh")}
    parts["Adjoint"] = adjoint[start:adjoint.index("\n};", start)]
    for name, text in parts.items():
        assert "__ldg" not in text, name
        assert not re.search(r"const\s+(S|T|float)\s*\*\s*__restrict__", text), name
