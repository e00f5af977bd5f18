"""The one-CTA FFT passes and the operator form's passes over the atoms' image rows, on
images whose baselines turn too fast per pixel for a smaller grid: sides 2048, 4096 and
8192."""
import functools
import math

import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance
SIDES = [(600, 2048), (1100, 4096), (2100, 8192)]


@functools.lru_cache(maxsize=None)
def _array(N, M, seed=0):
    """Baselines of up to 0.4 turns per pixel over four degrees, a few w-planes."""
    fov = math.radians(4.0)
    rng = np.random.default_rng(N + seed)
    uvw = rng.uniform(-1.0, 1.0, (M, 3)) * np.array([0.4 * N / fov, 0.4 * N / fov, 600.0])
    uvw[:4, :2] = np.array([[1, 1], [-1, 1], [1, -1], [-1, -1]]) * 0.4 * N / fov
    return fov, uvw


@pytest.mark.parametrize("coplanar", [False, True])
@pytest.mark.parametrize("N,G", SIDES)
def test_operators(N, G, coplanar):
    from paper_2406_01342_gb300 import abi
    fov, uvw = _array(N, 1500)
    if coplanar:
        uvw = uvw * np.array([1.0, 1.0, 0.0])
    M = uvw.shape[0]
    plan, stockham = abi.pc_plan_create(to_dev(uvw), N, fov), abi.pc_plan_create(to_dev(uvw), N, fov, fft_kernel=1)
    assert abi.pc_plan_transforms(plan) == dict(transform_grid=G, transform_image=N)
    assert abi.pc_plan_info(plan)["grid_side"] == G and abi.pc_plan_tuning_info(plan)["fft_warp"] == 3
    rng = np.random.default_rng(N)
    h = (rng.normal(size=M) + 1j * rng.normal(size=M)).astype(np.complex64)
    img = abi.pc_adjoint_grid(plan, to_dev(h)).cpu().numpy().ravel()
    border = np.concatenate([np.arange(N), (N - 1) * N + np.arange(N), np.arange(N) * N, np.arange(N) * N + N - 1])
    pix = np.union1d(border, rng.choice(N * N, 1500, replace=False))
    assert rel_l2(img[pix], operators.adjoint(uvw, N, fov, h.astype(np.complex128), pix)) <= TOL
    assert rel_l2(img, abi.pc_adjoint_grid(stockham, to_dev(h)).cpu().numpy().ravel()) <= TOL
    x = np.zeros(N * N, dtype=np.float32)
    x[pix] = rng.normal(size=pix.size)
    y = abi.pc_forward_grid(plan, to_dev(x.reshape(N, N))).cpu().numpy()
    assert rel_l2(y, operators.forward(uvw, N, fov, pix, x[pix].astype(np.float64))) <= TOL
    lhs = float(np.real(np.vdot(y.astype(np.complex128), h.astype(np.complex128))))
    rhs = float(np.sum(x.astype(np.float64) * img))
    assert abs(lhs - rhs) <= TOL * math.sqrt(float(np.sum(np.abs(y) ** 2) * np.sum(np.abs(h) ** 2)))


@pytest.mark.parametrize("N,G", SIDES)
def test_operator_form_matches_the_gram_form(N, G):
    """The operator pairs of the second form transform only the image rows that hold
    active atoms."""
    from paper_2406_01342_gb300 import abi
    fov, uvw = _array(N, 4000, 1)
    rng = np.random.default_rng(N + 1)
    at = np.sort(rng.choice(N * N, 12, replace=False))
    V = operators.forward(uvw, N, fov, at, rng.lognormal(0.0, 1.0, at.size))
    V = (V + 0.05 * (rng.normal(size=V.size) + 1j * rng.normal(size=V.size))).astype(np.complex64)
    plan = abi.pc_plan_create(to_dev(uvw), N, fov)
    assert abi.pc_plan_transforms(plan) == dict(transform_grid=G, transform_image=N)
    Vd = to_dev(V)
    lam = 0.2 * abi.pc_lambda_max(plan, Vd)
    a = abi.pc_solve(plan, Vd, lam, 0.01, reweight=1)
    b = abi.pc_solve(plan, Vd, lam, 0.01, reweight=2)
    assert a["converged"] and b["converged"] and a["idx"].numel() > 0
    assert a["idx"].cpu().numpy().tolist() == b["idx"].cpu().numpy().tolist()
    # the two forms stop on the relative change at 1e-5, from different step sizes
    assert abs(a["objective"] - b["objective"]) <= 1e-5 * a["objective"]
    xa, xb = a["x"].cpu().numpy().astype(np.float64), b["x"].cpu().numpy().astype(np.float64)
    assert abs(xa.sum() - xb.sum()) <= 1e-3 * abs(xa).sum()


@pytest.mark.parametrize("N,grid,image", [(600, 512, 256), (1100, 1024, 512)])
def test_transforms_of_short_baselines(N, grid, image):
    """And the smaller grid is named where it is used."""
    from paper_2406_01342_gb300 import abi
    fov, uvw = _array(N, 1500)
    plan = abi.pc_plan_create(to_dev(uvw * np.array([0.25, 0.25, 1.0])), N, fov)
    assert abi.pc_plan_transforms(plan) == dict(transform_grid=grid, transform_image=image)
    assert abi.pc_plan_info(plan)["grid_side"] == dict(SIDES)[N]
