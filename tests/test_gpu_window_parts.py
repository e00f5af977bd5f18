"""Window gridding and degridding with tiles split into small parts: few tiles, most of
the visibilities in the middle ones. The parts' size follows the slots, and the sums are
the direct ones."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance


@pytest.mark.parametrize("N,M,turns,spread", [(514, 300, 0.1, 1.0), (540, 20_000, 0.1, 0.2), (540, 60_000, 0.2, 0.01),
                                              (1100, 40_001, 0.08, 0.3), (300, 25_000, 0.2, 0.2)])
def test_parts(N, M, turns, spread):
    from paper_2406_01342_gb300 import abi
    fov = math.radians(3.5)
    rng = np.random.default_rng(M)
    r = np.minimum(np.abs(rng.normal(size=M)) * spread, 1.0) * turns * N / fov
    th = rng.uniform(0.0, 2.0 * math.pi, M)
    uvw = np.stack([r * np.cos(th), r * np.sin(th), rng.uniform(-1.0, 1.0, M) * 1000.0], axis=1)
    uvw[0, :2] = turns * N / fov, 0.0
    plan = abi.pc_plan_create(to_dev(uvw), N, fov, grid_mode=3)
    info, tune = abi.pc_plan_info(plan), abi.pc_plan_tuning_info(plan)
    assert tune["grid_mode"] == 3
    # a CTA's share of two on every SM (140 at least), and 16 slots a plane
    for piece in (tune["grid_piece"], tune["degrid_piece"]):
        assert 128 <= piece <= max(16 * info["n_planes"], info["n_slots"] / (2 * 140) + 1)
    k = np.sort(rng.choice(M, min(M, 3000), replace=False))
    h = np.zeros(M, dtype=np.complex64)
    h[k] = (rng.normal(size=k.size) + 1j * rng.normal(size=k.size)).astype(np.complex64)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    pix = np.union1d([0, N - 1, N * N - N, N * N - 1], rng.choice(N * N, 1500, replace=False))
    assert rel_l2(img[pix], operators.adjoint(uvw[k], N, fov, h[k].astype(np.complex128), pix)) <= TOL
    x = np.zeros(N * N, dtype=np.float32)
    x[pix] = rng.normal(size=pix.size)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    assert rel_l2(y[k], operators.forward(uvw[k], N, fov, pix, x[pix].astype(np.float64))) <= TOL
