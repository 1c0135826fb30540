"""Conversions of FP32 data, which run on sums of floats where those hold the values: the
exact result is rounded once; infinities, NaN and values at the ends of FP32's range come
out as in the FP64 form."""
from fractions import Fraction

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


def _rounded(x):
    """The float nearest to the rational x, ties to even."""
    y = np.float32(float(x))
    near = [y, np.nextafter(y, np.float32(np.inf)), np.nextafter(y, np.float32(-np.inf))]
    return min(near, key=lambda v: (abs(Fraction(float(v)) - x), int(v.view(np.uint32)) & 1))


def _state(buf, shape, ncomp):
    """The fields of a stored FP32 state, from its buffer (row pitch, ghosts and field order of the library)."""
    nx, ny, nz = shape
    al, g = (32, 1) if ncomp == 1 else (8, 2)
    px, py, nf = (nx + 16 + al - 1) // al * al, ny + 2 * g, 9 + ncomp
    fs, f = buf.numel() // nf, buf.cpu().numpy()
    f = f.reshape(fs // 32, nf, 32).transpose(1, 0, 2).reshape(nf, fs) if ncomp == 1 else f.reshape(nf, fs)
    return f[:, :nz * py * px].reshape(nf, nz, py, px)[:, :, g:g + ny, 8:8 + nx]


@pytest.mark.parametrize("ncomp", [1, 2])
@pytest.mark.parametrize("what", ["general", "equilibrium", "wide"])
def test_conversions_round_the_exact_result_once(ncomp, what):
    """Canonical float32 to state and back, against rational arithmetic; bit for bit."""
    shape = (11, 6, 5)
    nf, n = 9 + ncomp, 11 * 6 * 5
    m = inputs.random_moments(*shape, seed=9, nfields=nf).astype(np.float32).reshape(nf, n)
    r = np.random.default_rng(4)
    if what != "general":  # P near rho / 3, where A is what is left of it; densities and colours over a wide range
        if what == "wide":
            m[0] = r.uniform(0.01, 9.0, n)
            if ncomp == 2:
                m[1] = r.uniform(-0.01, 1.0, n) * 10.0 ** r.uniform(-9, 0, n)
        rho = m[:ncomp].astype(np.float64).sum(0)
        for f in range(ncomp + 3, ncomp + 6):
            m[f] = rho / 3 + r.choice([0.0, 1e-8, 1e-5, 1e-2], n) * r.normal(size=n)
    p = llb.llb_params_default(storage=llb.LLB_F32, ncomp=ncomp)
    size = llb.llb_state_bytes(*shape, 19, p) // 4
    bufs = [torch.zeros(size, dtype=torch.float32, device="cuda") for _ in range(2)]
    c = _ctx(shape, ncomp, llb.LLB_F32, bufs)
    try:
        llb.llb_init_moments_device(c, torch.from_numpy(m).cuda())
        out = torch.empty((nf, n), dtype=torch.float32, device="cuda")
        llb.llb_get_moments_device(c, out)
        llb.llb_synchronize(c)
        st = _state(bufs[0], shape, ncomp).reshape(nf, n)
    finally:
        llb.llb_destroy(c)
    out = out.cpu().numpy()
    ex = lambda a, i: Fraction(float(a[i]))  # noqa: E731
    for i in range(n):
        rho = ex(m[0], i) + (ex(m[1], i) if ncomp == 2 else 0)
        want = [rho - 1] + [ex(m[f], i) - (rho / 3 if f in range(ncomp + 3, ncomp + 6) else 0) for f in range(ncomp, nf)]
        for f, w in enumerate(want, ncomp - 1):
            assert st[f, i] == _rounded(w), ("state", f, i)
        rho = 1 + ex(st[ncomp - 1], i)
        want = ([ex(st[0], i), rho - ex(st[0], i)] if ncomp == 2 else [rho]) + \
            [ex(st[f], i) + (rho / 3 if f in range(ncomp + 3, ncomp + 6) else 0) for f in range(ncomp, nf)]
        for f, w in enumerate(want):
            assert out[f, i] == _rounded(w), ("canonical", f, i)
