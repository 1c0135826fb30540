"""Conversions of FP32 data, which run on pairs of floats where those hold the values:
infinities, NaN and values at the ends of FP32's range come out as in the FP64 form."""
import numpy as np
import pytest

from paper_2301_01622_gb300 import inputs, llb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [(1, llb.LLB_F32), (1, llb.LLB_F16S), (1, llb.LLB_BF16S), (2, llb.LLB_F32)]


def _ctx(shape, ncomp, storage, bufs=(None, None)):
    return llb.llb_create(*shape, 19, 0.8, llb.llb_params_default(ncomp=ncomp, storage=storage, buffers=bufs))


@pytest.mark.parametrize("ncomp, storage", CASES)
def test_values_a_pair_of_floats_cannot_hold(ncomp, storage):
    """Each canonical field in turn set to such a value at one node: what is infinite or NaN
    in the state and in what is read back does not depend on the type the values came in or
    go out as."""
    shape = (12, 5, 4)
    nf = 9 + ncomp
    m = torch.from_numpy(inputs.random_moments(*shape, seed=3, nfields=nf)).float()
    flat = m.view(nf, -1)
    for k, v in enumerate((np.inf, -np.inf, np.nan, 3e38, -3e38, 1e-30, 1e-42, 0.0)):
        for f in range(nf):
            flat[f, nf * k + f] = v
    if ncomp == 2:  # a total density beyond FP32's range
        flat[0, -1] = flat[1, -1] = 3e38
    out = []
    for dt in (torch.float32, torch.float64):
        c = _ctx(shape, ncomp, storage)
        try:
            llb.llb_init_moments_device(c, m.to("cuda", dt))
            got = [torch.empty(m.shape, dtype=t, device="cuda") for t in (torch.float32, torch.float64)]
            for g in got:
                llb.llb_get_moments_device(c, g)
            llb.llb_synchronize(c)
        finally:
            llb.llb_destroy(c)
        out.append([g.cpu().numpy() for g in got])
    (a32, a64), (b32, b64) = out
    assert np.isinf(b64).sum() > 10 and np.isnan(b64).sum() > 10
    with np.errstate(over="ignore"):
        pairs = ((a64, b64), (a32, a64.astype(np.float32)), (b32, b64.astype(np.float32)))
    for x, y in pairs:
        assert np.array_equal(np.isnan(x), np.isnan(y))
        assert np.array_equal(np.isinf(x), np.isinf(y)) and np.array_equal(x[np.isinf(x)], y[np.isinf(x)])
