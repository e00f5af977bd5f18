"""Tensor-core contraction at the edges of its tiles: 128-row tiles, column
chunks of 16 to 256, stages of 16 visibilities, one or several CTAs per tile."""
import numpy as np
import pytest

from oracle import operators
from tests.helpers import rel_l2, to_dev, workload

pytestmark = pytest.mark.gpu
TOL = 1e-5     # the operators' tolerance (three FP16 products hold 22 bits, FP32 accumulation)


@pytest.mark.parametrize("S,M", [(1, 7), (15, 16), (16, 17), (112, 2000), (127, 300), (128, 129), (129, 1000),
                                 (255, 500), (256, 2000), (257, 130), (384, 2000), (513, 1999), (1100, 700),
                                 (2400, 600)])
def test_gram_tile_edges(S, M):
    import torch  # noqa: F401
    from paper_2406_01342_gb300 import abi
    wl, V = workload("tiny_64_coplanar")
    uvw = np.ascontiguousarray(wl.uvw[:M])
    plan = abi.pc_plan_create(to_dev(uvw), wl.N, wl.fov)
    idx = np.sort(np.random.default_rng(S).choice(wl.N * wl.N, S, replace=False)).astype(np.int32)
    Vs = V[:M].astype(np.complex64)
    G, b = abi.pc_gram(plan, to_dev(Vs), to_dev(idx), mode=2)
    A = operators.phase_block(uvw, *operators.pixel_lmn(wl.N, wl.fov, idx))
    Gg = G.cpu().numpy()
    assert np.array_equal(Gg, Gg.T)
    assert rel_l2(Gg, np.real(A.conj().T @ A)) <= TOL
    assert rel_l2(b.cpu().numpy(), np.real(A.conj().T @ Vs.astype(np.complex128))) <= TOL
    G2, _ = abi.pc_gram(plan, None, to_dev(idx), mode=2)      # without the V column
    assert rel_l2(G2.cpu().numpy(), Gg) <= TOL
