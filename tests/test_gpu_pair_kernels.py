"""The kernels that hold two nodes per thread, at the sizes where their tiles end:
boxes smaller than a tile and than its halo, exact multiples of a tile, one more
and one less, against the FP64 oracle; and the periodic ghost copies they keep.
FP32 bound: 1e-5 per moment group, as in the other FP32 parity tests."""
import numpy as np
import pytest

from oracle import D3Q19, D3Q27, lb
from oracle import two_component as tc
from paper_2301_01622_gb300 import inputs, llb

from gpu_helpers import GROUPS_2, assert_fields, assert_groups, run_gpu

pytestmark = pytest.mark.gpu

LAT = {19: D3Q19, 27: D3Q27}

# tiles of the one-component kernel: 30 x 6 outputs
SHAPES_1 = [(1, 1, 1), (2, 3, 1), (5, 4, 3), (15, 2, 4), (16, 7, 2), (29, 5, 4), (30, 6, 5), (31, 7, 3), (61, 13, 6),
            (90, 18, 4)]


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("shape", SHAPES_1, ids=lambda s: "x".join(map(str, s)))
def test_one_component_tile_edges(shape, q):
    """Random moments, 3 steps, also as one graph (the steps before the last write no ghost copies)."""
    m0 = inputs.random_moments(*shape, seed=7 + shape[0] + 3 * shape[1])
    ref = lb.run_moment_only(m0, LAT[q], 0.7, 3)
    ctx = llb.llb_create(*shape, q, 0.7, llb.llb_params_default(storage=llb.LLB_F32))
    try:
        got = np.empty_like(m0)
        for step in (llb.llb_step, llb.llb_step_graph):
            llb.llb_init_moments(ctx, m0)
            step(ctx, 3)
            llb.llb_get_moments(ctx, got)
            assert_groups(got, ref, 1e-5, what=f"{shape} D3Q{q} {step.__name__}")
    finally:
        llb.llb_destroy(ctx)


# One step from the same stored state: the two kernels differ by FP32 rounding, so a
# stored element may fall on the other side of a rounding boundary: one spacing of the
# storage format, 2^-10 (FP16) or 2^-7 (BF16) of the largest element, and the FP32 bound.
@pytest.mark.parametrize("storage, ulp", [(llb.LLB_F16S, 2.0**-10), (llb.LLB_BF16S, 2.0**-7)], ids=["f16", "bf16"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (5, 4, 3), (31, 7, 3), (60, 13, 6)], ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("q", [19, 27])
def test_one_component_narrow_storage(shape, q, storage, ulp):
    m0 = inputs.random_moments(*shape, seed=11)
    a, _ = run_gpu(shape, q, 0.7, 1, m0=m0, storage=storage, kernel=llb.LLB_KERNEL_TILED)
    b, _ = run_gpu(shape, q, 0.7, 1, m0=m0, storage=storage, kernel=llb.LLB_KERNEL_DIRECT)
    assert_fields(a, b, ulp + 1e-5, what=f"{shape} D3Q{q}")


@pytest.mark.parametrize("storage", [llb.LLB_F32, llb.LLB_F16S, llb.LLB_BF16S], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", [(1, 1, 2), (5, 3, 2), (15, 7, 4), (16, 1, 3), (47, 13, 5)],
                         ids=lambda s: "x".join(map(str, s)))
def test_one_component_ghost_copies(shape, storage):
    """Every ghost position of the state holds the node it mirrors, bit for bit."""
    import torch

    nx, ny, nz = shape
    p = llb.llb_params_default(storage=storage)
    es = 4 if storage == llb.LLB_F32 else 2
    n = llb.llb_state_bytes(nx, ny, nz, 19, p) // es
    bufs = [torch.zeros(n, dtype=torch.int32 if es == 4 else torch.int16, device="cuda") for _ in range(2)]
    ctx = llb.llb_create(nx, ny, nz, 19, 0.8, llb.llb_params_default(storage=storage, buffers=bufs))
    try:
        llb.llb_init_moments(ctx, inputs.random_moments(nx, ny, nz, seed=3))
        llb.llb_step(ctx, 3)
        llb.llb_synchronize(ctx)
    finally:
        llb.llb_destroy(ctx)
    al = 32 if es == 4 else 8
    px, py, gx = (nx + 16 + al - 1) // al * al, ny + 2, 8
    fs, f = n // 10, bufs[1].cpu().numpy()
    f = f.reshape(fs // 32, 10, 32).transpose(1, 0, 2).reshape(10, fs) if es == 4 else f.reshape(10, fs)
    f = f[:, :nz * py * px].reshape(10, nz, py, px)
    core = f[:, :, 1:1 + ny, 8:8 + nx]
    # a box narrower than the ghost columns copies each node once per side
    gx = min(gx, nx)
    ys, xs = np.arange(-1, ny + 1), np.arange(-gx, nx + gx)
    want = core[:, :, ys % ny][:, :, :, xs % nx]
    assert np.array_equal(f[:, :, :, 8 + xs[0]:8 + xs[-1] + 1], want)


# tiles of the two-component kernel: 28 x 10 outputs
SHAPES_2 = [(4, 4, 4), (15, 6, 5), (16, 11, 4), (28, 10, 6), (29, 9, 4), (27, 21, 7), (57, 20, 5), (84, 31, 4)]


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("shape", SHAPES_2, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("eps", [0.0, 0.02], ids=["sharp", "smooth"])
def test_two_component_tile_edges(shape, q, eps):
    """Random moments (an interface normal at every node), 2 steps."""
    nx, ny, nz = shape
    m0 = inputs.random_moments(nx, ny, nz, seed=5 + nx + 3 * ny, nfields=11)
    prm = tc.CGParams(beta=0.6, A_s=0.03, g_min=1e-6, eps=eps)
    ref = tc.run_moment_only(m0, LAT[q], 0.8, prm, 2)
    got, _ = run_gpu(shape, q, 0.8, 2, m0=m0, storage=llb.LLB_F32, ncomp=2, beta=0.6, A_s=0.03, g_min=1e-6, grad_eps=eps)
    assert_groups(got, ref, 1e-5, GROUPS_2, what=f"{shape} D3Q{q}")


@pytest.mark.parametrize("h_c", [0, 1, 3, 5])
def test_two_component_probe_ranges(h_c):
    """Every probe range of the near-contact detector, both nodes of a pair and the
    wrap in each direction: a droplet pair two nodes apart across the box's faces."""
    shape = (33, 24, 17)
    r1, r2, u = inputs.droplets(*shape, [(5.3, 11.6, 1.2), (27.4, 12.9, 1.7)], [4.6, 4.6], [(-0.02, 0, 0), (0.02, 0, 0)])
    tot = np.concatenate([r1[None], r2[None], (r1 + r2) * u, np.stack([u[a] * u[b] + (a == b) / 3 for a, b in
                          ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])])
    prm = tc.CGParams(A_h=0.02, h_c=h_c, g_min=1e-6)
    ref = tc.run_moment_only(tot, D3Q19, 0.9, prm, 2)
    got, _ = run_gpu(shape, 19, 0.9, 2, m0=tot, storage=llb.LLB_F32, ncomp=2, A_h=0.02, h_c=h_c, g_min=1e-6)
    assert_groups(got, ref, 1e-5, GROUPS_2, what=f"h_c={h_c}")


@pytest.mark.parametrize("shape", [(5, 4, 4), (15, 7, 4), (40, 23, 5)], ids=lambda s: "x".join(map(str, s)))
def test_two_component_ghost_copies(shape):
    """Every ghost position of the state holds the node it mirrors, bit for bit."""
    import torch

    nx, ny, nz = shape
    p = llb.llb_params_default(storage=llb.LLB_F32, ncomp=2)
    n = llb.llb_state_bytes(nx, ny, nz, 27, p) // 4
    bufs = [torch.zeros(n, dtype=torch.float32, device="cuda") for _ in range(2)]
    p = llb.llb_params_default(storage=llb.LLB_F32, ncomp=2, buffers=bufs)
    ctx = llb.llb_create(nx, ny, nz, 27, 0.8, p)
    try:
        llb.llb_init_moments(ctx, inputs.random_moments(nx, ny, nz, seed=3, nfields=11))
        llb.llb_step(ctx, 3)
        llb.llb_synchronize(ctx)
    finally:
        llb.llb_destroy(ctx)
    px, py, gx, gy = (nx + 16 + 7) // 8 * 8, ny + 4, min(8, nx), 2
    fs = n // 11
    f = bufs[1].cpu().numpy().reshape(11, fs)[:, :nz * py * px].reshape(11, nz, py, px)
    core = f[:, :, 2:2 + ny, 8:8 + nx]
    ys, xs = np.arange(-gy, ny + gy), np.arange(-gx, nx + gx)
    want = core[:, :, ys % ny][:, :, :, xs % nx]
    assert np.array_equal(f[:, :, 2 + ys[0]:2 + ys[-1] + 1, 8 + xs[0]:8 + xs[-1] + 1], want)
