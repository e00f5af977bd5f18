"""Transforms on a smaller image where the w-term makes up much of a visibility's
turns: its slope is steepest beyond the image's border, where the interpolation's outer
taps lie. Turns per pixel just under a limit of the rule (forty taps on a grid of 512 or
1024), as a band without that slope would have it. Adjoint and forward against the direct sum, on the border and inside."""
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
# the operators on the image's own grid leave 1e-6 over an image, up to three times that
# on its border (the kernel's correction is largest there); the interpolation 4e-7
TOL = 4e-6


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("N,fov_deg,turns,share,w_lo", [
    (600, 30.0, 0.137, 0.2, 0.97), (600, 30.0, 0.137, 0.5, 0.97), (600, 30.0, 0.137, 0.9, 0.97), (600, 30.0, 0.137, 0.5, -1.0),
    (1100, 12.0, 0.163, 0.2, 0.97), (1100, 12.0, 0.163, 0.5, 0.97), (1100, 12.0, 0.071, 0.9, 0.97),
    (2048, 20.0, 0.04, 0.2, 0.97), (2048, 20.0, 0.04, 0.5, 0.97), (2048, 20.0, 0.04, 0.9, 0.97)])
def test_small_image_with_a_large_w_term(N, fov_deg, turns, share, w_lo, sign):
    from paper_2406_01342_gb300 import abi
    fov, M = math.radians(fov_deg), 600
    half = 0.5 * fov
    rng = np.random.default_rng(N)
    # most of the baselines at the ends of the range: u, v = +-(1 - share) turns per pixel
    uv = (1.0 - share) * turns * N / fov
    w = share * turns * N / fov * math.sqrt(1.0 - 2.0 * half * half) / half
    uvw = np.stack([uv * rng.choice([-1.0, 1.0], M) * rng.uniform(0.97, 1.0, M),
                    uv * rng.choice([-1.0, 1.0], M) * rng.uniform(0.97, 1.0, M),
                    sign * w * rng.uniform(w_lo, 1.0, M)], axis=1)
    plan = abi.pc_plan_create(to_dev(uvw), N, fov, max_planes=1024)
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    border = np.unique(np.concatenate([np.arange(N), (N - 1) * N + np.arange(N), np.arange(N) * N,
                                       np.arange(N) * N + N - 1]))
    ref = operators.adjoint(uvw, N, fov, h.astype(np.complex128), border)
    assert rel_l2(img[border], ref) <= TOL
    pix = np.union1d(border, rng.choice(N * N, 1000, replace=False))
    x = np.zeros(N * N, dtype=np.float32)
    x[pix] = rng.normal(size=pix.size)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    assert rel_l2(y, operators.forward(uvw, N, fov, pix, x[pix].astype(np.float64))) <= TOL
