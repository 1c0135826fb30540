"""Conversions and reductions that carry pairs of floats in place of FP64 (FP32
inputs and states): against the FP64 path of the same calls."""
import numpy as np
import pytest

from paper_2301_01622_gb300 import inputs, llb

pytestmark = pytest.mark.gpu

CASES = [(1, llb.LLB_F32), (1, llb.LLB_F16S), (1, llb.LLB_BF16S), (2, llb.LLB_F32)]


def _ctx(shape, ncomp, storage):
    return llb.llb_create(*shape, 19, 0.8, llb.llb_params_default(ncomp=ncomp, storage=storage))


@pytest.mark.parametrize("ncomp, storage", CASES)
@pytest.mark.parametrize("shape", [(4, 4, 4), (33, 7, 5), (65, 40, 9)], ids=lambda s: "x".join(map(str, s)))
def test_conversions_match_the_fp64_path(shape, ncomp, storage):
    """The same values as float32 and as float64, in and out: both sides round the
    exact result once, so they agree to one unit in the last place of float32."""
    m = inputs.random_moments(*shape, seed=11, nfields=9 + ncomp).astype(np.float32)
    out = []
    for x in (m, m.astype(np.float64)):
        c = _ctx(shape, ncomp, storage)
        try:
            llb.llb_init_moments(c, x)
            out.append([llb.llb_get_moments(c, np.empty(m.shape, t)) for t in (np.float32, np.float64)])
        finally:
            llb.llb_destroy(c)
    ulp = np.spacing(np.abs(out[1][1]).astype(np.float32))
    # the 16-bit state: a last-place difference of the float can move the stored value by one of its own steps
    state = {llb.LLB_F32: 0.0, llb.LLB_F16S: 2.0 ** -10, llb.LLB_BF16S: 2.0 ** -7}[storage]
    lim = ulp + state * np.abs(out[1][1] - (1.0 if ncomp == 1 else 0.0))
    assert np.all(np.abs(out[0][1] - out[1][1]) <= lim)  # in
    for a, b in out:
        assert np.all(np.abs(a.astype(np.float64) - b) <= ulp)  # out


@pytest.mark.parametrize("ncomp, storage", CASES)
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 4, 4), (70, 33, 9)], ids=lambda s: "x".join(map(str, s)))
def test_diagnostics_match_fp64_sums(shape, ncomp, storage):
    """Sums of the stored moments; rounding bound 1e-12 of the sum of magnitudes."""
    if ncomp == 2 and min(shape) < 4:
        pytest.skip("two components need 4 nodes per direction")
    m = inputs.random_moments(*shape, seed=5, nfields=9 + ncomp, rho_spread=0.6)
    c = _ctx(shape, ncomp, storage)
    try:
        llb.llb_init_moments(c, m)
        got = llb.llb_diagnostics(c)
        x = llb.llb_get_moments(c, np.empty(m.shape))
    finally:
        llb.llb_destroy(c)
    rho = x[0] if ncomp == 1 else x[0] + x[1]
    drop, j, n = x[0], x[ncomp:ncomp + 3], rho.size
    inside = drop > 0.5
    assert abs(got["mass"][0] - drop.sum()) <= 1e-12 * n
    assert ncomp == 1 or abs(got["mass"][1] - x[1].sum()) <= 1e-12 * n
    assert np.all(np.abs(np.array(got["momentum"]) - j.sum((1, 2, 3))) <= 1e-12 * n)
    assert got["n_in"] == int(inside.sum()) and abs(got["rho1_sum"] - drop[inside].sum()) <= 1e-12 * n
    assert abs(got["min_rho"] - rho.min()) <= 1e-12 and got["flags"] == 0


def test_diagnostics_flag_and_keep_what_is_not_finite():
    """A NaN or an infinity in one node sets the flag and spoils its own sum alone."""
    import torch

    for bad, value in ((1, np.nan), (0, np.inf), (7, np.inf)):
        m = torch.from_numpy(inputs.random_moments(20, 9, 5, seed=2)).float().cuda()
        m[bad, 2, 3, 4] = value
        d = llb.llb_diagnostics_noalloc(m, 20, 9, 5)
        assert d["flags"] & llb.LLB_FLAG_NONFINITE and np.isnan(d["min_rho"])
        assert np.isfinite(d["momentum"][1]) and np.isfinite(d["momentum"][2])
        assert np.isfinite(d["momentum"][0]) == (bad != 1)
        assert d["mass"][0] == np.inf if bad == 0 else np.isfinite(d["mass"][0])
