"""Sparse forward operator over its kernels: few and many visibilities and
atoms, w-terms of none to many turns (fixed-point and double-float phases)."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance


@pytest.mark.parametrize("M,S,N,fov_deg,w_max", [
    (1, 1, 16, 1.0, 0.0), (33, 7, 64, 12.0, 40.0), (2000, 1025, 64, 1.0, 0.0), (39_999, 9, 512, 2.0, 1.2e4),
    (40_001, 12, 512, 2.0, -300.0), (100_003, 33, 2048, 5.0, 4000.0), (400_001, 5, 512, 5.0, 1.6e4),
    (1_000_001, 3, 4096, 5.0, 4200.0), (5000, 40, 256, 30.0, 2000.0), (5000, 40, 256, 60.0, 0.0)])
def test_forward_sparse_over_sizes_and_w(M, S, N, fov_deg, w_max):
    from paper_2406_01342_gb300 import abi
    fov = math.radians(fov_deg)
    rng = np.random.default_rng(M + S)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([0.3 * N / fov, 0.3 * N / fov, 0.5 * abs(w_max)])
    uvw[:, 2] += 0.5 * w_max                       # w from 0 to w_max
    idx = np.sort(rng.choice(N * N, S, replace=False)).astype(np.int32)
    x = rng.lognormal(0.0, 1.0, S).astype(np.float32) * rng.choice([-1.0, 1.0], S).astype(np.float32)
    plan = abi.pc_plan_create(to_dev(uvw), N, fov, max_planes=4096)
    y = abi.pc_forward_sparse(plan, to_dev(idx), to_dev(x)).cpu().numpy()
    k = rng.choice(M, min(M, 4000), replace=False)
    assert rel_l2(y[k], operators.forward(uvw[k], N, fov, idx, x.astype(np.float64))) <= TOL
