"""What FP32 rounding does to the colour density adds up from step to step where the fluid
is uniform: inside a droplet in motion it is the same in every step."""
import numpy as np
import pytest

from oracle import lb
from paper_2301_01622_gb300 import inputs, llb

from gpu_helpers import run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", [19, 27])
@pytest.mark.parametrize("speed", [0.03, 0.0401, 0.0453, 0.05, 0.0557, 0.0603])
def test_rounding_of_a_moving_droplet_does_not_add_up(speed, q):
    """FP32 against FP64, 30 steps: rho1 in the 2-norm within 2^-22, four halves of a unit in
    the last place of 1 (30 steps that round the same way would be 30 of them)."""
    n = 64
    r1, r2, u = inputs.droplets(n, n, n, [(n / 2, n / 2, n / 2)], [20.0], [(speed, 0, 0)])
    m0 = np.concatenate([r1[None], r2[None], lb.equilibrium_moments(r1 + r2, u)[1:]]).astype(np.float32).astype(np.float64)
    got = [run_gpu((n, n, n), q, 1.0, 30, m0=m0, storage=s, ncomp=2, A_h=0.01)[0] for s in (llb.LLB_F64, llb.LLB_F32)]
    assert np.linalg.norm(got[1][0] - got[0][0]) <= 2.0**-22 * np.linalg.norm(got[0][0])
