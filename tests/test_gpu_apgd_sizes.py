"""The restricted LASSO at the edges of its kernels' ranges (rows per warp, groups
of 32 rows, columns per thread, rows of a cluster's CTAs, rows in shared memory and
read from L2; aligned and unaligned rows of G) against the same problem solved in
64 bits."""
import numpy as np
import pytest

from tests.helpers import to_dev

pytestmark = pytest.mark.gpu


def solve64(G, b, lam, positive):
    L = np.linalg.eigvalsh(G)[-1]
    x = y = np.zeros_like(b)
    t = 1.0
    for _ in range(2000):
        u = y - (G @ y - b) / L
        z = np.maximum((u if positive else np.abs(u)) - lam / L, 0.0)
        z = z if positive else np.copysign(z, u)
        t1 = 0.5 * (1.0 + np.sqrt(1.0 + 4.0 * t * t))
        if np.dot(y - z, z - x) > 0.0:      # restart: linear convergence
            t, t1, y = 1.0, 1.0, z
        else:
            y = z + (t - 1.0) / t1 * (z - x)
        done = np.linalg.norm(z - x) <= 1e-13 * np.linalg.norm(z)
        x, t = z, t1
        if done:
            break
    return x


# A Wishart matrix of 4 n draws: condition about 9, so that the stop (1e-6 of the
# iterate) and the FP32 products leave about 9 (1e-6 + 6e-8 sqrt(n)) <= 4e-5
@pytest.mark.parametrize("positive", [False, True])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 96, 127, 128, 129, 192, 193, 223, 224, 225, 260, 513, 850,
                               898, 901, 904, 1303, 1700, 2497, 2800])
def test_apgd_at_the_edges(n, positive):
    import torch

    from paper_2406_01342_gb300 import abi
    rng = np.random.default_rng(n)
    A = rng.normal(size=(4 * n, n))
    G = A.T @ A
    b = G @ np.where(rng.random(n) < 0.5, rng.normal(size=n), 0.0) + 0.1 * n ** 0.5 * rng.normal(size=n)
    lam = 0.1 * float(np.abs(b).max())
    ref = solve64(G.astype(np.float32).astype(np.float64), b.astype(np.float32).astype(np.float64), lam, positive)
    x = torch.zeros(n, dtype=torch.float32, device="cuda")
    x, it, _ = abi.pc_apgd(to_dev(G.astype(np.float32)), to_dev(b.astype(np.float32)), lam, 1e-6, 5000, x, positive=positive)
    assert it < 5000
    assert np.linalg.norm(x.cpu().numpy() - ref) <= 4e-5 * max(np.linalg.norm(ref), 1e-30)
