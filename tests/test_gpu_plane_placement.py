"""The w-planes' number, spacing and place against the direct sum where the range of
w is next to a whole number of spacings, far from zero, or hardly a range at all."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance


@pytest.mark.parametrize("offset", [0.0, -2500.0])
@pytest.mark.parametrize("spacings,N", [(1e-9, 64), (0.3, 64), (0.999, 256), (1.0, 64), (1.001, 512), (1.5, 256), (1.99, 300),
                                        (2.0, 64), (2.01, 128), (8.0, 64), (9.5, 512), (3.7, 1000)])
def test_adjoint_and_forward(spacings, N, offset):
    from paper_2406_01342_gb300 import abi
    fov, M = math.radians(4.0), 1200
    r2 = 0.5 * fov * fov
    dw = 1.0 / (2.0 * r2 / (1.0 + math.sqrt(1.0 - r2)))      # the widest spacing
    rng = np.random.default_rng(N)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([0.25 * N / fov, 0.25 * N / fov, 0.5 * spacings * dw])
    uvw[0, 2], uvw[1, 2] = -0.5 * spacings * dw, 0.5 * spacings * dw
    uvw[:, 2] += offset
    plan = abi.pc_plan_create(to_dev(uvw), N, fov)
    info = abi.pc_plan_info(plan)
    assert info["kernel_width"] < info["n_planes"] <= math.ceil(spacings * 1.4) + info["kernel_width"]
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    pix = np.union1d([0, N - 1, N * N - N, N * N - 1], rng.choice(N * N, 1500, replace=False))
    assert rel_l2(img[pix], operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)) <= TOL
    x = np.zeros(N * N, dtype=np.float32)
    x[pix] = rng.normal(size=pix.size)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    assert rel_l2(y, operators.forward(uvw, N, fov, pix, x[pix].astype(np.float64))) <= TOL
