"""dL/domega of FP32 states: its sums are as accurate as FP64's and have its range."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2301_01622_gb300 import build as B
from paper_2301_01622_gb300 import inputs, llb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def sum_terms(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("terms")
    exe = str(d / "adjoint_terms_check")
    r = subprocess.run([nvcc, *B.ARCH, "-O3", "-std=c++17", "-I", B.CSRC, os.path.join(ROOT, "tests", "adjoint_terms_check.cu"),
                        "-o", exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]

    def run(a, b, r, c):
        path = str(d / "terms.bin")
        with open(path, "wb") as f:
            f.write(np.int32(len(a)).tobytes())
            f.write(np.concatenate([a, b, r[:, None], c], axis=1).astype(np.float32).tobytes())
        p = subprocess.run([exe, path], capture_output=True, text=True, timeout=60)
        assert p.returncode == 0, (p.returncode, p.stderr)
        return float.fromhex(p.stdout.strip()) if p.stdout.strip() not in ("inf", "-inf", "nan", "-nan") else float(p.stdout)

    return run


def _terms(case, n, g):
    """a, b, r, c of n nodes: the sizes of a flow, b r close to c, and the ends of the ranges."""
    a = g.normal(size=(n, 6))
    b = 1e-3 * g.normal(size=(n, 6)) ** 2
    r = 1.0 + 0.05 * g.normal(size=n)
    c = 1e-3 * g.normal(size=(n, 6))
    if case in ("close", "cancelling"):
        c = (b * r[:, None]) * (1.0 + 1e-6 * g.normal(size=(n, 6)))
    if case == "cancelling":  # the sum itself cancels: nodes again with the opposite sign, in another order
        h = n // 2
        k = g.permutation(h)
        a[h:2 * h], b[h:2 * h], r[h:2 * h], c[h:2 * h] = -a[k], b[k], r[k], c[k]
    if case == "small":
        a *= 2.0**-110
    if case == "tiny":
        b, c = b * 2.0**-100, c * 2.0**-100
    if case == "large":
        a, b, c = a * 2.0**70, b * 2.0**40, c * 2.0**40
    if case == "mixed":  # nodes of every size side by side
        a *= 2.0 ** g.integers(-120, 100, size=(n, 1))
    if case == "zeros":
        a[::3] = 0.0
        b[1::3], c[1::3] = 0.0, 0.0
    return [v.astype(np.float32) for v in (a, b, r, c)]


@pytest.mark.parametrize("case", ["flow", "close", "cancelling", "small", "tiny", "large", "mixed", "zeros"])
def test_terms_against_rational_arithmetic(sum_terms, case):
    """Error at most one rounding of the sum to FP64 and 2^-58 of the sum of magnitudes (FP64
    itself would be held to 2^-53 of it for every term of a thread, 200 here); nodes that run
    in FP64 are held to FP64's bound."""
    n = 1024
    a, b, r, c = _terms(case, n, np.random.default_rng(7))
    got = sum_terms(a, b, r, c)
    ex = mag = Fraction(0)
    for i in range(n):
        ri = Fraction(float(r[i]))
        for k in range(6):
            x, y, z = (Fraction(float(v[i, k])) for v in (a, b, c))
            ex += x * (y * ri - z)
            mag += abs(x) * (abs(y * ri) + abs(z))
    wide = case in ("small", "tiny", "large", "mixed")
    lim = abs(ex) * Fraction(1, 2**52) + mag * (Fraction(200, 2**53) if wide else Fraction(1, 2**58))
    assert abs(Fraction(got) - ex) <= lim


def test_terms_that_are_not_finite(sum_terms):
    a, b, r, c = _terms("flow", 64, np.random.default_rng(8))
    c[5, 2] = np.inf
    a[5, 2] = 1.0
    assert sum_terms(a, b, r, c) == -np.inf
    c[40, 0] = np.nan
    assert np.isnan(sum_terms(a, b, r, c))


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("ncomp", [1, 2])
def test_dtau_beyond_the_range_of_float(ncomp, q):
    """Finite cotangents whose terms add up to more than 3.4e38: against FP64 states, to the
    1e-4 of the other FP32 gradients."""
    shape = (40, 9, 6)
    nf = 9 + ncomp
    m = inputs.random_moments(*shape, seed=5, nfields=nf)
    m[ncomp + 3:ncomp + 6] += 3.0  # A = 3, so every term is about as large as its cotangent
    g = np.zeros_like(m)
    g[ncomp + 3:ncomp + 6] = 3e36 * (1.0 + 0.1 * np.random.default_rng(1).normal(size=(3,) + m.shape[1:]))
    res = []
    for storage, dt in ((llb.LLB_F64, torch.float64), (llb.LLB_F32, torch.float32)):
        gd = torch.from_numpy(g).to("cuda", dt)
        gi = torch.empty_like(gd)
        two = dict(ncomp=2, grad_eps=0.05) if ncomp == 2 else {}
        c = llb.llb_create(*shape, q, 0.8, llb.llb_params_default(storage=storage, **two))
        try:
            llb.llb_init_moments(c, m)
            res.append(llb.llb_adjoint(c, 1, gd, gi))
        finally:
            llb.llb_destroy(c)
    assert abs(res[0]) > 3.5e38 and np.isfinite(res[1])
    assert abs(res[1] - res[0]) <= 1e-4 * abs(res[0])
