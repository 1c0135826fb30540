"""A device wait of the two-component step that cannot complete (its barrier is armed for
a byte that never arrives; the copies themselves land) runs out after its bound, is
reported as LLB_ETIMEOUT by the calls that synchronise and leaves the CUDA context usable."""
import numpy as np
import pytest

from oracle import D3Q19, lb
from oracle import two_component as tc
from paper_2301_01622_gb300 import inputs, llb

pytestmark = pytest.mark.gpu

SHAPE = (64, 40, 24)
STUCK = dict(ncomp=2, storage=llb.LLB_F32, wait_budget_ms=20, debug_flags=1)


def _drop(shape):
    nx, ny, nz = shape
    r1, r2, u = inputs.droplets(nx, ny, nz, [(nx / 2, ny / 2, nz / 2)], [min(shape) / 4], [(0.02, 0, 0)])
    return np.concatenate([r1[None], r2[None], lb.equilibrium_moments(r1 + r2, u)[1:]])


def _status(fn, *args):
    with pytest.raises(llb.LLBError) as e:
        fn(*args)
    return e.value.status


def _device_still_works():
    shape = (20, 12, 8)
    m0 = _drop(shape)
    ctx = llb.llb_create(*shape, 19, 0.9, llb.llb_params_default(storage=llb.LLB_F32, ncomp=2))
    try:
        llb.llb_init_moments(ctx, m0)
        llb.llb_step(ctx, 2)
        got = llb.llb_get_moments(ctx, np.empty_like(m0))
    finally:
        llb.llb_destroy(ctx)
    ref = tc.run_moment_only(m0, D3Q19, 0.9, tc.CGParams(g_min=1e-6), 2)
    assert np.abs(got - ref).max() < 1e-5


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("graph", [False, True], ids=["step", "graph"])
def test_single_box_reports_the_timeout(q, graph):
    m0 = _drop(SHAPE)
    for read in (llb.llb_synchronize, lambda c: llb.llb_get_moments(c, np.empty_like(m0)), llb.llb_diagnostics):
        ctx = llb.llb_create(*SHAPE, q, 0.9, llb.llb_params_default(**STUCK))
        try:
            llb.llb_init_moments(ctx, m0)
            (llb.llb_step_graph if graph else llb.llb_step)(ctx, 2)
            assert _status(read, ctx) == llb.LLB_ETIMEOUT
            assert _status(llb.llb_step, ctx, 1) == llb.LLB_ESTATE  # sticky from now on
        finally:
            llb.llb_destroy(ctx)
    _device_still_works()


def test_host_step_reports_the_timeout():
    m0 = _drop(SHAPE)
    ctx = llb.llb_create(*SHAPE, 19, 0.9, llb.llb_params_default(**STUCK))
    try:
        assert _status(llb.llb_step_host, ctx, m0, np.empty_like(m0), 2) == llb.LLB_ETIMEOUT
    finally:
        llb.llb_destroy(ctx)
    _device_still_works()


@pytest.mark.parametrize("graph", [False, True], ids=["step", "graph"])
def test_every_box_of_a_batch_reports_the_timeout(graph):
    """More boxes than CTAs: a CTA whose wait has given up goes on to items of other boxes,
    and each of those has to report that its step was not done."""
    dims = [(8, 6, 5)] * 700  # one item each; at most four CTAs on each of up to 160 SMs
    b = llb.llb_batch_create(dims, 19, 0.9, llb.llb_params_default(**STUCK))
    try:
        m0 = _drop(dims[0])
        for k in range(len(dims)):
            llb.llb_init_moments(llb.llb_batch_domain(b, k), m0)
        (llb.llb_batch_step_graph if graph else llb.llb_batch_step)(b, 1)
        got = [_status(llb.llb_synchronize, llb.llb_batch_domain(b, k)) for k in range(len(dims))]
        assert got == [llb.LLB_ETIMEOUT] * len(dims)
    finally:
        llb.llb_batch_destroy(b)
    _device_still_works()


@pytest.mark.parametrize("params", [dict(STUCK, grad_eps=0.05), dict(storage=llb.LLB_F32, kernel=llb.LLB_KERNEL_TMA,
                                    wait_budget_ms=20, debug_flags=1)], ids=["two-component", "one-component-tma"])
def test_adjoint_reports_the_timeout(params):
    """The forward steps of a gradient wait too, and the call synchronises."""
    import torch

    m0 = _drop(SHAPE)
    if params.get("ncomp", 1) == 1:
        m0 = np.concatenate([m0[:1] + m0[1:2], m0[2:]])
    g = torch.ones(m0.shape, dtype=torch.float32, device="cuda")
    ctx = llb.llb_create(*SHAPE, 19, 0.9, llb.llb_params_default(**params))
    try:
        llb.llb_init_moments(ctx, m0)
        assert _status(llb.llb_adjoint, ctx, 4, g, torch.empty_like(g)) == llb.LLB_ETIMEOUT
        assert _status(llb.llb_step, ctx, 1) == llb.LLB_ESTATE
    finally:
        llb.llb_destroy(ctx)
    _device_still_works()


def test_autotuners_report_the_timeout():
    """Their trials run the kernel that waits, and they synchronise."""
    c = llb.llb_create(*SHAPE, 19, 0.9, llb.llb_params_default(**STUCK))
    try:
        llb.llb_init_moments(c, _drop(SHAPE))
        assert _status(llb.llb_autotune, c, 1) == llb.LLB_ETIMEOUT
        assert _status(llb.llb_step, c, 1) == llb.LLB_ESTATE
    finally:
        llb.llb_destroy(c)
    b = llb.llb_batch_create([(8, 6, 5), (16, 9, 7)], 19, 0.9, llb.llb_params_default(**STUCK))
    try:
        for k, d in enumerate([(8, 6, 5), (16, 9, 7)]):
            llb.llb_init_moments(llb.llb_batch_domain(b, k), _drop(d))
        assert _status(llb.llb_batch_autotune, b, 1) == llb.LLB_ETIMEOUT
        assert _status(llb.llb_batch_step, b, 1) == llb.LLB_ESTATE
    finally:
        llb.llb_batch_destroy(b)
    _device_still_works()
