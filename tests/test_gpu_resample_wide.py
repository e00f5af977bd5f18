"""The transpose of the interpolation where its bands are widest: large images of short
baselines, which the smallest grid and forty taps sample. Forward and adjoint against the
direct sum."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance


@pytest.mark.parametrize("N,turns", [(4096, 0.0197), (3522, 0.0228)])
def test_widest_bands(N, turns):
    from paper_2406_01342_gb300 import abi
    fov, M = math.radians(3.0), 300
    rng = np.random.default_rng(N)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([turns * N / fov, turns * N / fov, 1.0])
    uvw[0, :2] = turns * N / fov
    plan = abi.pc_plan_create(to_dev(uvw), N, fov)
    pix = np.union1d([0, N - 1, N * N - N, N * N - 1], rng.choice(N * N, 3000, replace=False))
    x = np.zeros(N * N, dtype=np.float32)
    x[pix] = rng.normal(size=pix.size)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    assert rel_l2(y, operators.forward(uvw, N, fov, pix, x[pix].astype(np.float64))) <= TOL
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    assert rel_l2(img[pix], operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)) <= TOL
