"""Coplanar gridding and the shared-memory FFT at the smallest sizes: few
visibilities to a CTA, one row to a CTA, odd counts, against the direct sum."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M", [(16, 1), (16, 33), (30, 257), (64, 2000), (100, 31), (128, 5003), (250, 64), (514, 700)])
@pytest.mark.parametrize("kw", [{}, {"kernel_width": 8}, {"kernel_width": 4}])
def test_coplanar_adjoint(N, M, kw):
    from paper_2406_01342_gb300 import abi
    fov = math.radians(1.5)
    rng = np.random.default_rng(N + M)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([0.4 * N / fov, 0.4 * N / fov, 0.0])
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    plan = abi.pc_plan_create(to_dev(uvw), N, fov, **kw)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    pix = np.arange(N * N) if N <= 128 else np.sort(rng.choice(N * N, 3000, replace=False))
    ref = operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)
    # the operators' tolerance; a kernel of four cells aliases 1000 times as much as one of seven
    assert rel_l2(img[pix], ref) <= (5e-3 if kw.get("kernel_width") == 4 else 1e-5)
