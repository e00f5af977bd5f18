"""The sparse forward operator's error against 64 bits at the edges of its kinds of phase
(few atoms and visibilities: full FP32 sines; then angles of 31 bits, then of 23)."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [3000, 99_999, 100_001, 1_000_100])
@pytest.mark.parametrize("S", [1, 10, 16, 17, 256, 257])
def test_error(M, S):
    from paper_2406_01342_gb300 import abi
    N, fov = 256, math.radians(4.0)
    rng = np.random.default_rng(S)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([0.2 * N / fov, 0.2 * N / fov, 0.1 * N / fov])
    idx = np.sort(rng.choice(N * N, S, replace=False)).astype(np.int32)
    x = rng.lognormal(0.0, 1.0, S).astype(np.float32)
    plan = abi.pc_plan_create(to_dev(uvw), N, fov)
    y = abi.pc_forward_sparse(plan, to_dev(idx), to_dev(x)).cpu().numpy()
    k = np.sort(rng.choice(M, 3000, replace=False))
    ref = operators.forward(uvw[k], N, fov, idx, x.astype(np.float64))
    # the lattice phases' rounding (2^-33 turns times half the side, both axes) leaves
    # 5e-8 rad, the FP32 turns 5e-8, sine and products 6e-8, a sum of 16 terms 1e-7;
    # beyond, angles to 2^-25 turns add 1.1e-7 and longer sums up to 3e-7
    assert rel_l2(y[k], ref) <= (1.6e-7 if S <= 16 and M < 100_000 else 4e-7)
