"""Adjoint and forward far from w = 0, against the direct sum: n - 1 enters with |w| turns,
so its own accuracy shows."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance; float64 sums leave 2 pi 1e9 1e-16 of it


@pytest.mark.parametrize("w_off", [1e7, -1e9])
@pytest.mark.parametrize("N,fov_deg,w_range", [(128, 2.0, 0.0), (256, 5.0, 3000.0), (512, 12.0, 200.0)])
def test_far_from_zero(N, fov_deg, w_range, w_off):
    from paper_2406_01342_gb300 import abi
    fov, M = math.radians(fov_deg), 700
    rng = np.random.default_rng(N)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([0.3 * N / fov, 0.3 * N / fov, 0.5 * w_range])
    uvw[:, 2] += w_off
    plan = abi.pc_plan_create(to_dev(uvw), N, fov)
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    pix = np.union1d([0, N - 1, N * N - N, N * N - 1], rng.choice(N * N, 1500, replace=False))
    assert rel_l2(img[pix], operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)) <= TOL
    x = np.zeros(N * N, dtype=np.float32)
    x[pix] = rng.normal(size=pix.size)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    assert rel_l2(y, operators.forward(uvw, N, fov, pix, x[pix].astype(np.float64))) <= TOL
