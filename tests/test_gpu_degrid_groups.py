"""Degridding over plane groups at the edges of its groups and pieces: eight planes (two
groups of four) to two dozen, one visibility, a piece and one more, several pieces of a
tile, against the direct sum."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance


@pytest.mark.parametrize("M", [1, 127, 129, 257, 3000, 170_001])
@pytest.mark.parametrize("spacings", [0.0, 0.5, 2.5, 5.5, 6.5, 16.2])
def test_forward(M, spacings):
    from paper_2406_01342_gb300 import abi
    N, fov = 96, math.radians(4.0)
    r2 = 0.5 * fov * fov
    dw = 1.0 / (2.0 * r2 / (1.0 + math.sqrt(1.0 - r2)))
    rng = np.random.default_rng(M)
    # three clusters of baselines: a few heavy tiles
    c = rng.uniform(-0.3, 0.3, (3, 2))[rng.integers(0, 3, M)] + 0.01 * rng.normal(size=(M, 2))
    uvw = np.concatenate([c * N / fov, rng.uniform(-0.5, 0.5, (M, 1)) * spacings * dw], axis=1)
    uvw[0, 2] = -0.5 * spacings * dw
    uvw[-1, 2] = 0.5 * spacings * dw
    plan = abi.pc_plan_create(to_dev(uvw), N, fov)
    x = rng.normal(size=N * N).astype(np.float32)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    k = np.union1d([0, M - 1], rng.integers(0, M, 400))
    assert rel_l2(y[k], operators.forward(uvw[k], N, fov, np.arange(N * N), x.astype(np.float64))) <= TOL
