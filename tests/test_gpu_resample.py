"""Transforms on a smaller image: adjoint and forward against the direct sum
at the image's border and inside, on the edges of the rule (turns per pixel, a
w-term, sides that are no power of two), and the adjoint identity between them."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance


@pytest.mark.parametrize("N,turns,fov_deg,w_max,kw", [
    (514, 0.40, 2.0, 1500.0, {}), (640, 0.10, 3.0, 700.0, {}), (1000, 0.30, 2.0, 0.0, {}), (1026, 0.33, 4.0, 300.0, {}),
    (1100, 0.27, 5.0, 600.0, {"grid_mode": 2}), (1100, 0.05, 12.0, 120.0, {"autotune": 1}),
    (2048, 0.145, 5.0, 1000.0, {}), (2050, 0.08, 2.0, 0.0, {}), (600, 0.02, 30.0, 20.0, {}),
    (600, 0.10, 30.0, -40.0, {"max_planes": 14})])
def test_small_image_transforms(N, turns, fov_deg, w_max, kw):
    from paper_2406_01342_gb300 import abi
    fov, M = math.radians(fov_deg), 1500
    rng = np.random.default_rng(N)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([turns * N / fov, turns * N / fov, 0.5 * abs(w_max)])
    uvw[:4, :2] = np.array([[1, 1], [-1, 1], [1, -1], [-1, -1]]) * turns * N / fov
    uvw[:, 2] += 0.5 * w_max
    plan = abi.pc_plan_create(to_dev(uvw), N, fov, **kw)
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    border = np.concatenate([np.arange(N), (N - 1) * N + np.arange(N), np.arange(N) * N, np.arange(N) * N + N - 1])
    pix = np.union1d(border, rng.choice(N * N, 2000, replace=False))
    assert rel_l2(img[pix], operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)) <= TOL
    assert abi.pc_lambda_max(plan, to_dev(h)) == float(np.abs(img).max())
    x = np.zeros(N * N, dtype=np.float32)
    x[pix] = rng.normal(size=pix.size)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    ref = operators.forward(uvw, N, fov, pix, x[pix].astype(np.float64))
    assert rel_l2(y, ref) <= TOL
    lhs = float(np.real(np.vdot(y.astype(np.complex128), h.astype(np.complex128))))
    rhs = float(np.sum(x.astype(np.float64) * img))
    assert abs(lhs - rhs) <= TOL * math.sqrt(float(np.sum(np.abs(y) ** 2) * np.sum(np.abs(h) ** 2)))
