"""The second FFT pass where the number of warps per image row changes (just past a wave of
rows; eight to twelve planes and more), against the direct sum on every row."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance


@pytest.mark.parametrize("N", [304, 306, 322, 324])
@pytest.mark.parametrize("spacings", [0.5, 2.5, 5.5, 9.5])
def test_adjoint(N, spacings):
    from paper_2406_01342_gb300 import abi
    fov, M = math.radians(4.0), 900
    r2 = 0.5 * fov * fov
    dw = 1.0 / (2.0 * r2 / (1.0 + math.sqrt(1.0 - r2)))
    rng = np.random.default_rng(N)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([0.3 * N / fov, 0.3 * N / fov, 0.5 * spacings * dw])
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    plan = abi.pc_plan_create(to_dev(uvw), N, fov)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy()
    cols = rng.integers(0, N, (N, 5))
    pix = np.unique((np.arange(N)[:, None] * N + cols).ravel())
    assert rel_l2(img.ravel()[pix], operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)) <= TOL
    assert abi.pc_lambda_max(plan, to_dev(h)) == float(np.abs(img).max())
