"""A box whose rows are longer than 2^31 elements of the interleaved FP32 state
(220,000,000 x 2 x 1: 35 GB per state copy): the step writes the periodic ghost copies
where they belong and nothing else."""
import numpy as np
import pytest

from oracle import D3Q19, lb
from paper_2301_01622_gb300 import inputs, llb

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NX, NY, TAU = 220_000_000, 2, 0.8


def test_ghost_copies_of_rows_beyond_2_31_elements():
    p = llb.llb_params_default(storage=llb.LLB_F32)
    n = llb.llb_state_bytes(NX, NY, 1, 19, p) // 4
    need = 10 * NX * NY * 4 + 2 * 4 * n
    free, _ = torch.cuda.mem_get_info()
    if free < need * 1.1:
        pytest.skip(f"needs {need / 1e9:.0f} GB of device memory, {free / 1e9:.0f} GB free")
    rng = np.random.default_rng(5)
    xs = [0, 1, 7, 8, NX - 9, NX - 8, NX - 1] + [int(v) for v in rng.integers(0, NX, 20)]
    # inner nodes that a distance cut to 32 bits (2^32 elements short, 2^32 / 10 nodes) would reach
    px = (NX + 16 + 31) // 32 * 32
    for first in (px + NX - 2**32 // 10, 2**32 // 10 - px - 8):
        assert 0 <= first < NX - 16
        xs += list(range(first - 8, first + 16))
    m = inputs.random_moments_device(NX, NY, 1, seed=3)
    bufs = [torch.zeros(n, dtype=torch.float32, device="cuda") for _ in range(2)]
    ctx = llb.llb_create(NX, NY, 1, 19, TAU, llb.llb_params_default(storage=llb.LLB_F32, buffers=bufs))
    try:
        before = {}
        for x in xs:
            ix = torch.tensor([(x - 1) % NX, x, (x + 1) % NX], device="cuda")
            for y in range(NY):
                iy = torch.tensor([(y - 1) % NY, y, (y + 1) % NY], device="cuda")
                v = m[:, 0][:, iy[:, None], ix[None, :]].double().cpu().numpy()
                before[x, y] = np.repeat(v[:, None], 3, axis=1)  # one plane: its own neighbour in z
        llb.llb_init_moments_device(ctx, m)
        llb.llb_step(ctx, 1)
        llb.llb_get_moments_device(ctx, m)
        llb.llb_synchronize(ctx)
        for (x, y), nb in before.items():
            ref = lb.node_moment_only(nb, D3Q19, TAU, 1, 1, 1)
            got = m[:, 0, y, x].double().cpu().numpy()
            assert np.abs(got - ref).max() <= 1e-6, (x, y)

        # ghost columns and rows of the stored state, bit for bit
        def at(x, y):
            i = (y + 1) * px + x + 8
            return (i // 32 * 32) * 10 + i % 32 + 32 * torch.arange(10, device="cuda")[:, None]

        ends = torch.cat([torch.arange(-8, 8, device="cuda"), torch.arange(NX - 8, NX + 8, device="cuda")])
        for y in range(-1, NY + 1):
            a, b = bufs[1][at(ends, y)], bufs[1][at(ends % NX, y % NY)]
            assert torch.equal(a, b), y
    finally:
        llb.llb_destroy(ctx)
        del m, bufs
        torch.cuda.empty_cache()
