"""Dirty images of coplanar arrays are as close to 64 bits as the image's own grid gives
them (fft_kernel = 1 always transforms on it), also where that oversamples more than twice."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,turns", [(514, 0.1), (700, 0.2), (1100, 0.05)])
def test_error_is_that_of_the_own_grid(N, turns):
    from paper_2406_01342_gb300 import abi
    fov, M = math.radians(3.0), 3000
    rng = np.random.default_rng(N)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([turns * N / fov, turns * N / fov, 0.0])
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    pix = np.sort(rng.choice(N * N, 4000, replace=False))
    ref = operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)
    err = [rel_l2(abi.pc_adjoint_grid(abi.pc_plan_create(to_dev(uvw), N, fov, fft_kernel=k), to_dev(h))
                  .cpu().numpy().ravel()[pix], ref) for k in (0, 1)]
    # the two runs differ in the order of the grid's sums and in the passes' last bits
    assert err[0] <= 1.1 * err[1]
