"""Diagnostics of FP32 data: the sums are as accurate as FP64's and have its range."""
import math

import numpy as np
import pytest

from paper_2301_01622_gb300 import inputs, llb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rest(shape):
    m = np.zeros((10,) + shape[::-1], dtype=np.float32)
    m[0] = 1.0
    m[4:7] = np.float32(1 / 3)
    return m


def _both(m, shape):
    """llb_diagnostics of an FP32 state and llb_diagnostics_noalloc of the float32 moments."""
    dev = torch.from_numpy(np.ascontiguousarray(m)).cuda()
    c = llb.llb_create(*shape, 19, 0.8, llb.llb_params_default(storage=llb.LLB_F32))
    try:
        llb.llb_init_moments_device(c, dev)
        return [llb.llb_diagnostics(c), llb.llb_diagnostics_noalloc(dev, *shape)]
    finally:
        llb.llb_destroy(c)


def test_sums_keep_what_fp64_keeps():
    """1 + 2^-25 + 2^-51 fits FP64 and no pair of floats, whichever nodes and threads hold the terms."""
    shape = (70, 9, 3)
    want = 1.0 + 2.0**-25 + 2.0**-51
    for at in ((0, 1, 2), (5, 800, 40), (1889, 0, 900)):
        m = _rest(shape)
        for a in (1, 2, 3):
            m[a].reshape(-1)[list(at)] = [1.0, 2.0**-25, 2.0**-51]
        for d in _both(m, shape):
            assert list(d["momentum"]) == [want] * 3


def test_like_terms_and_cancelling_terms():
    """FP64's own bound for the terms of a thread and the tree above it: 64 x 2^-53 of the
    sum of magnitudes (at most 64 terms a thread in these boxes)."""
    shape = (128, 96, 80)
    n = 128 * 96 * 80
    m = inputs.random_moments(*shape, seed=6).astype(np.float32)
    m[1] = np.float32(0.9)                     # like terms
    m[2] = np.random.default_rng(2).normal(size=m[2].shape)
    m[2].reshape(-1)[n // 2:] = -m[2].reshape(-1)[:n // 2][::-1]  # cancels to nothing
    for d in _both(m, shape):
        for a in (1, 2, 3):
            v = m[a].astype(np.float64).reshape(-1)
            assert abs(d["momentum"][a - 1] - math.fsum(v)) <= 64 * 2.0**-53 * np.abs(v).sum()


def test_sums_beyond_the_range_of_float():
    """Finite data whose sums leave FP32's range: FP64 holds them."""
    shape = (40, 5, 4)
    m = _rest(shape)
    m[1] = 3e38
    m[2, 0, 0, :8] = 3e38
    m[2, 1, 0, :8] = -3e38
    m[0, 3] = 2e38
    for d in _both(m, shape):
        assert d["flags"] == 0
        assert d["momentum"][0] == pytest.approx(800 * float(np.float32(3e38)), rel=1e-12)
        assert d["momentum"][1] == 0.0 and d["momentum"][2] == 0.0
        assert d["mass"][0] == pytest.approx(200 * float(np.float32(2e38)), rel=1e-6)


def test_two_components_beyond_the_range_of_float():
    shape = (16, 6, 5)
    m = np.concatenate([_rest(shape)[:1], _rest(shape)])
    m[0], m[1] = 0.25, 0.75
    m[2] = -3e38
    m[0, 1:3] = 1e38
    c = llb.llb_create(*shape, 19, 0.8, llb.llb_params_default(storage=llb.LLB_F32, ncomp=2))
    try:
        llb.llb_init_moments_device(c, torch.from_numpy(m).cuda())
        d = llb.llb_diagnostics(c)
    finally:
        llb.llb_destroy(c)
    n, big = 480, 192 * float(np.float32(1e38))
    assert d["flags"] == 0 and d["n_in"] == 192
    assert d["momentum"][0] == pytest.approx(-n * float(np.float32(3e38)), rel=1e-12)
    assert d["rho1_sum"] == pytest.approx(big, rel=1e-12) and d["mass"][0] == pytest.approx(big, rel=1e-12)
