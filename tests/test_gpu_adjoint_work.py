"""llb_adjoint over the step kernels and its working memory: kernels that take any
pair of state buffers (states stepped in place) and kernels tied to the context's own
(states copied) give one gradient and leave the state as it was, in the library's
memory and in the caller's."""
import numpy as np
import pytest

from paper_2301_01622_gb300 import inputs, llb

pytestmark = pytest.mark.gpu

SHAPE = (48, 13, 9)
CASES = [(llb.LLB_KERNEL_TILED, 0), (llb.LLB_KERNEL_TILED, 1), (llb.LLB_KERNEL_TMA, 2), (llb.LLB_KERNEL_DIRECT, 0)]


def _grad(kernel, variant, storage, steps, every, give):
    import torch

    nx, ny, nz = SHAPE
    dt = torch.float64 if storage == llb.LLB_F64 else torch.float32
    m0 = inputs.random_moments(nx, ny, nz, seed=2)
    g = torch.from_numpy(np.random.default_rng(5).uniform(-1, 1, m0.shape)).to("cuda", dt)
    gi = torch.empty_like(g)
    p = llb.llb_params_default(storage=storage, kernel=kernel, variant=variant if storage == llb.LLB_F32 else 0)
    c = llb.llb_create(nx, ny, nz, 19, 0.8, p)
    try:
        llb.llb_init_moments(c, m0)
        before = llb.llb_get_moments(c, np.empty_like(m0))
        n = llb.llb_adjoint_bytes(c, steps, every)
        work = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda") if give else None
        dtau = llb.llb_adjoint(c, steps, g, gi, every=every, work=work)
        assert np.array_equal(before, llb.llb_get_moments(c, np.empty_like(m0)))
        if give:
            with pytest.raises(llb.LLBError):
                llb.llb_adjoint(c, steps, g, gi, every=every, work=work[:n - 1])
    finally:
        llb.llb_destroy(c)
    return gi.double().cpu().numpy(), dtau


@pytest.mark.parametrize("storage, tol", [(llb.LLB_F64, 1e-12), (llb.LLB_F32, 1e-5)], ids=["f64", "f32"])
@pytest.mark.parametrize("steps, every", [(0, 0), (1, 0), (7, 1), (7, 3), (6, 3), (7, 20)])
def test_step_kernels_and_working_memory(steps, every, storage, tol):
    ref, rtau = _grad(llb.LLB_KERNEL_DIRECT, 0, llb.LLB_F64, steps, 1, False)
    for kernel, variant in CASES:
        for give in (False, True):
            got, dtau = _grad(kernel, variant, storage, steps, every, give)
            assert np.abs(got - ref).max() <= tol * np.abs(ref).max(), (kernel, variant, give)
            assert abs(dtau - rtau) <= 10 * tol * max(abs(rtau), 1.0), (kernel, variant, give)


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 1), (5, 4, 3), (29, 5, 4), (30, 6, 5), (31, 7, 3), (61, 13, 4)],
                         ids=lambda s: "x".join(map(str, s)))
def test_fp32_adjoint_tile_edges(shape, q):
    """The FP32 adjoint (tiles of 30 x 6, two nodes per thread) against the FP64 one
    (one node per thread), 3 steps.  FP32 bound 1e-5 of the largest entry, as above."""
    import torch

    nx, ny, nz = shape
    m0 = inputs.random_moments(nx, ny, nz, seed=4)
    g64 = torch.from_numpy(np.random.default_rng(6).uniform(-1, 1, m0.shape)).to("cuda")
    out = []
    for storage, dt in ((llb.LLB_F64, torch.float64), (llb.LLB_F32, torch.float32)):
        g = g64.to(dt)
        gi = torch.empty_like(g)
        c = llb.llb_create(nx, ny, nz, q, 0.7, llb.llb_params_default(storage=storage))
        try:
            llb.llb_init_moments(c, m0)
            dtau = llb.llb_adjoint(c, 3, g, gi)
        finally:
            llb.llb_destroy(c)
        out.append((gi.double().cpu().numpy(), dtau))
    (a, ta), (b, tb) = out
    assert np.abs(a - b).max() <= 1e-5 * np.abs(a).max()
    assert abs(ta - tb) <= 1e-4 * max(abs(ta), 1.0)


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("shape", [(4, 4, 4), (33, 5, 7), (32, 8, 4), (31, 9, 8)], ids=lambda s: "x".join(map(str, s)))
def test_two_component_adjoint_does_not_see_the_tiles(shape, q):
    """A box shifted along its diagonal has the shifted gradient: where tiles and runs of
    planes begin must not show.  FP64, 2 steps: 1e-11 of the largest entry (the sums of
    a node are the same, in another order)."""
    import torch

    nx, ny, nz = shape
    m0 = inputs.random_moments(nx, ny, nz, seed=8, nfields=11)
    g0 = np.random.default_rng(9).uniform(-1, 1, m0.shape)
    c = llb.llb_create(nx, ny, nz, q, 0.9, llb.llb_params_default(storage=llb.LLB_F64, ncomp=2, grad_eps=0.05))
    out = []
    try:
        for shift in ((0, 0, 0), (1, 2, 3)):
            g = torch.from_numpy(np.ascontiguousarray(np.roll(g0, shift, axis=(1, 2, 3)))).cuda()
            gi = torch.empty_like(g)
            llb.llb_init_moments(c, np.ascontiguousarray(np.roll(m0, shift, axis=(1, 2, 3))))
            dtau = llb.llb_adjoint(c, 2, g, gi)
            out.append((np.roll(gi.cpu().numpy(), [-s for s in shift], axis=(1, 2, 3)), dtau))
    finally:
        llb.llb_destroy(c)
    (a, ta), (b, tb) = out
    assert np.abs(a - b).max() <= 1e-11 * np.abs(a).max()
    assert abs(ta - tb) <= 1e-10 * max(abs(ta), 1.0)
