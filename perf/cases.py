"""The calls whose speed is kept an eye on: what a user of the library has it
do, from the smallest operator call to the 4096 x 4096 solve.

A case names an entry point ("op"), the image side N, the visibility count M,
the array (stations within radius_m metres of a centre, Earth rotation at 100
MHz, field of view fov_deg) and what the call takes besides (S atoms, sources).
The arrays, skies and noise follow paper_2406_01342_gb300/synth.py, drawn on
the GPU so that ten million visibilities take a moment. Visibilities are made
from the sky by a direct sum in torch, never by the library's own operators.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2406_01342_gb300 import abi

WAVELENGTH = 2.99792458           # metres at 100 MHz
LAT = math.radians(-30.0)
DEC = math.radians(-30.0)


def _case(name, op, N, M, fov_deg=2.0, stations=40, radius_m=3000.0, sources=50, S=0, coplanar=False):
    return dict(name=name, op=op, N=N, M=M, fov_deg=fov_deg, stations=stations, radius_m=radius_m,
                sources=sources, S=S, coplanar=coplanar)


def listed():
    return [
        # a dirty image of the smallest configuration (64 x 64, w = 0): what a call costs by itself
        _case("dirty_64", "dirty", 64, 2000, 1.0, 0, 0.0, 5, coplanar=True),
        # adjoint onto a four-scale dictionary, shaped like the diffuse experiment (256 x 256, 251 stations)
        _case("dict_256", "dict", 256, 31600, 6.5, 251, 900.0, 40),
        # one dual certificate of a Frank-Wolfe iteration, the ordinary size (512 x 512, 200k)
        _case("certificate_512", "certificate", 512, 200_000, S=50),
        # a one-off image: new baselines, so plan and dirty image in one go; a side that is no power of two
        _case("snapshot_1100", "snapshot", 1100, 123_457, 5.0, 60, 5000.0, 100),
        # model visibilities of a dense image (degridding), 2048 x 2048
        _case("forward_2048", "forward", 2048, 2_000_000, 5.0, 60, 5000.0, 200),
        # one dual certificate of the largest configuration
        _case("certificate_4096", "certificate", 4096, 10_000_000, 5.0, 100, 5850.0, 500, S=500),
        # a contraction over many visibilities, ragged in both
        _case("gram_1001", "gram", 2048, 1_000_003, 5.0, 60, 5000.0, 200, S=1001),
        # model visibilities of a sparse image (the residual of an iteration)
        _case("sparse_629", "sparse", 2048, 2_000_000, 5.0, 60, 5000.0, 200, S=629),
        # the restricted LASSO: a late active set, and the first one of a 512 x 512 solve
        _case("apgd_120", "apgd", 512, 20_000, S=120),
        _case("apgd_1300", "apgd", 512, 20_000, S=1300),
        # whole solves: the ordinary one, and a request of the serving stream's larger kind
        _case("solve_512", "solve", 512, 200_000),
        _case("solve_1024", "solve", 1024, 500_000, 5.0, 60, 5000.0, 100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another call over the same ranges: image sides 64..4096, 2k..10M
    visibilities, arrays whose longest baseline turns 0.08 to 0.28 times per
    pixel at the image's edge of resolution (as the configurations' arrays do)."""
    op = rng.choice(["dirty", "dict", "certificate", "certificate", "snapshot", "forward", "forward",
                     "gram", "gram", "sparse", "apgd", "solve"])
    # the ranges of each call: image side, visibilities, atoms
    n_lo, n_hi, m_lo, m_hi, s_lo, s_hi = {
        "dirty": (64, 4096, 2_000, 10_000_000, 0, 0),
        "dict": (64, 1024, 2_000, 300_000, 0, 0),
        "certificate": (128, 4096, 10_000, 10_000_000, 5, 500),
        "snapshot": (128, 2048, 10_000, 2_000_000, 0, 0),
        "forward": (64, 4096, 2_000, 10_000_000, 0, 0),
        "gram": (256, 2048, 20_000, 1_000_000, 65, 1100),
        "sparse": (256, 2048, 10_000, 2_000_000, 5, 1000),
        "apgd": (512, 512, 20_000, 20_000, 20, 2500),
        "solve": (256, 1024, 10_000, 1_000_000, 0, 0),
    }[op]
    t = rng.random()                       # images and visibility counts grow together, loosely
    near = min(1.0, max(0.0, t + rng.uniform(-0.15, 0.15)))
    N = 2 * int(round(math.exp(math.log(n_lo) + t * math.log(n_hi / n_lo)) / 2))
    M = int(round(math.exp(math.log(m_lo) + near * math.log(m_hi / m_lo))))
    fov_deg = round(rng.uniform(1.0, 6.5), 2)
    # past 512 x 512 the fields are those of the configurations, so that the number of w-planes is too
    if N > 512:
        fov_deg = round(rng.uniform(2.0, 5.0), 2)
    turns = rng.uniform(0.08, 0.28)
    radius = turns * N / math.radians(fov_deg) * WAVELENGTH / 2.0
    stations = rng.randint(40, 100)
    K = _log(rng, 5, 200)
    return dict(op=op, N=N, M=M, fov_deg=fov_deg, stations=stations, radius_m=round(radius, 1), sources=K,
                S=_log(rng, s_lo, s_hi) if s_hi else 0, coplanar=op == "dirty" and rng.random() < 0.25)


# ---------------------------------------------------------------- inputs


def _generator(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + stream)
    return g


def _uvw(case, seed):
    """(M, 3) float64 wavelengths on the GPU, in time order."""
    M, dev = case["M"], "cuda"
    g = _generator(seed, 1)

    def rand(*n):
        return torch.rand(*n, generator=g, device=dev, dtype=torch.float64)

    if case["coplanar"]:
        # Gaussian-radial coverage of a disk that reaches the finest scale the pixels hold
        R = 0.5 * case["N"] / math.radians(case["fov_deg"])
        if case["radius_m"]:
            R = 2.0 * case["radius_m"] / WAVELENGTH
        r = torch.randn(M, generator=g, device=dev, dtype=torch.float64).abs() * (R / 2.0)
        r = torch.where(r > R, R * rand(M), r)
        th = 2.0 * math.pi * rand(M)
        return torch.stack([r * torch.cos(th), r * torch.sin(th), torch.zeros_like(r)], dim=1)
    n = case["stations"]
    r = case["radius_m"] * torch.sqrt(rand(n))
    th = 2.0 * math.pi * rand(n)
    east, north = r * torch.cos(th), r * torch.sin(th)
    ij = torch.triu_indices(n, n, 1, device=dev)
    X = -math.sin(LAT) * (north[ij[1]] - north[ij[0]])
    Y = east[ij[1]] - east[ij[0]]
    Z = math.cos(LAT) * (north[ij[1]] - north[ij[0]])
    n_b = X.numel()
    # four hours symmetric about transit; M of the (dump, baseline) pairs
    n_t = max(360, -(-M // n_b))
    dump_s = 4.0 * 3600.0 / n_t
    pick = torch.randperm(n_t * n_b, generator=g, device=dev)[:M].sort().values
    H = ((pick // n_b).double() - (n_t - 1) / 2.0) * (dump_s * 2.0 * math.pi / 86164.0905)
    X, Y, Z = X[pick % n_b], Y[pick % n_b], Z[pick % n_b]
    sH, cH, sd, cd = torch.sin(H), torch.cos(H), math.sin(DEC), math.cos(DEC)
    return torch.stack([sH * X + cH * Y, -sd * cH * X + sd * sH * Y + cd * Z,
                        cd * cH * X - cd * sH * Y + sd * Z], dim=1) / WAVELENGTH


def _pixels(case, seed, stream, n):
    """n distinct pixels in raster order (int64)."""
    N = case["N"]
    return torch.randperm(N * N, generator=_generator(seed, stream), device="cuda")[:n].sort().values


def _directions(case, idx):
    """(3, S) direction cosines l, m, n - 1 and (S,) n of raster indices, float64."""
    N, fov = case["N"], math.radians(case["fov_deg"])
    l = ((idx // N).double() - N / 2) * (fov / N)
    m = ((idx % N).double() - N / 2) * (fov / N)
    n = torch.sqrt(1.0 - l * l - m * m)
    return torch.stack([l, m, -(l * l + m * m) / (1.0 + n)]), n


def _visibilities(case, seed, uvw):
    """Log-normal point sources seen by the array with 20 dB of noise: complex64 (M,), pixels, fluxes."""
    g = _generator(seed, 3)
    idx = _pixels(case, seed, 2, case["sources"])
    flux = torch.exp(torch.randn(idx.numel(), generator=g, device="cuda"))
    d, n = _directions(case, idx)
    M = uvw.shape[0]
    V = torch.empty(M, dtype=torch.complex64, device="cuda")
    amp = flux / n.float()
    step = max(1, 200_000_000 // max(1, idx.numel()))
    for a in range(0, M, step):
        t = uvw[a:a + step] @ d
        t -= torch.round(t)
        t = t.float() * (-2.0 * math.pi)
        V[a:a + step] = torch.complex(torch.cos(t) @ amp, torch.sin(t) @ amp)
    sigma = math.sqrt(float((V.real ** 2 + V.imag ** 2).mean()) * 10.0 ** -2.0)
    noise = torch.randn(M, 2, generator=g, device="cuda") * (sigma / math.sqrt(2.0))
    return V + torch.view_as_complex(noise), idx, flux


def _dense_image(case, seed):
    """An extended sky: a few Gaussian blobs over faint structure, N x N float32."""
    N, g = case["N"], _generator(seed, 4)
    at = torch.linspace(-1.0, 1.0, N, device="cuda")
    img = 0.01 * torch.rand(N, N, generator=g, device="cuda")
    p = torch.rand(10, 4, generator=g, device="cuda")
    for k in range(10):
        wx, wy = 0.005 + 0.05 * p[k, 2], 0.005 + 0.05 * p[k, 3]
        img += torch.exp(-((at[:, None] - 1.6 * p[k, 0] + 0.8) / wx) ** 2) * torch.exp(
            -((at[None, :] - 1.6 * p[k, 1] + 0.8) / wy) ** 2)
    return img


def _atoms(case, seed):
    """S active pixels as an exploration leaves them: lobes of neighbours around the brightest places."""
    S, N = case["S"], case["N"]
    centres = _pixels(case, seed, 5, max(1, S // 12))
    offs = torch.tensor([[i, j] for i in range(-2, 3) for j in range(-2, 3)], device="cuda")
    ij = torch.stack([centres // N, centres % N], dim=1)[:, None, :] + offs[None, :, :]
    ij = ij.clamp(0, N - 1).reshape(-1, 2)
    near = (ij[:, 0] * N + ij[:, 1]).unique()
    near = near[torch.randperm(near.numel(), generator=_generator(seed, 6), device="cuda")[:S]]
    return near.sort().values


def _support(case, seed, idx, flux):
    """S atoms of an iteration under way: the sources at most of their flux, then faint ones elsewhere."""
    S = case["S"]
    more = _pixels(case, seed, 5, S)
    at = torch.cat([idx[:S], more[~torch.isin(more, idx)][:max(0, S - idx.numel())]])
    x = torch.cat([0.8 * flux[:S], torch.full((at.numel(),), 0.05, device="cuda")])[:at.numel()]
    order = at.argsort()
    return at[order], x[order].contiguous()


def _dictionary():
    return abi.make_dictionary((0.0, 2.0, 5.0, 8.0))


def prepare(case, seed):
    op, fov = case["op"], math.radians(case["fov_deg"])
    uvw = _uvw(case, seed)
    st = dict(op=op, N=case["N"], fov=fov)
    if op == "apgd":
        # Gram matrix and right-hand side of an active set, as float32 contractions leave them
        idx = _atoms(case, seed)
        V, _, _ = _visibilities(case, seed, uvw)
        G, b = _contract(case, uvw, V, idx)
        st.update(G=G.float().contiguous(), b=b.float().contiguous(), lam=0.1 * float(b.abs().max()))
        return st
    if op == "forward":
        st.update(img=_dense_image(case, seed))
    elif op == "gram":
        V, _, _ = _visibilities(case, seed, uvw)
        st.update(V=V, idx=_atoms(case, seed).int())
    elif op == "sparse":
        idx = _pixels(case, seed, 5, case["S"])
        st.update(idx=idx.int(), x=torch.exp(torch.randn(idx.numel(), generator=_generator(seed, 6), device="cuda")))
    else:
        V, idx, flux = _visibilities(case, seed, uvw)
        st.update(V=V)
        if op == "certificate":
            at, x = _support(case, seed, idx, flux)
            st.update(idx=at.int(), x=x, lam=0.1 * case["M"] * float(flux.max()))
        elif op == "solve":
            # lambda = 0.1 lambda_max; near the brightest source's flux times M when sources do not overlap
            st.update(lam=0.1 * case["M"] * float(flux.max()))
    if op == "snapshot":
        st.update(uvw=uvw)
        return st
    st.update(plan=abi.pc_plan_create(uvw, case["N"], fov))
    return st


def run(state):
    op = state["op"]
    if op == "dirty":
        return abi.pc_adjoint_grid(state["plan"], state["V"])
    if op == "snapshot":
        plan = abi.pc_plan_create(state["uvw"], state["N"], state["fov"])
        return abi.pc_adjoint_grid(plan, state["V"])
    if op == "dict":
        return abi.pc_dict_adjoint(state["plan"], _dictionary(), state["V"])
    if op == "certificate":
        mu, mu_inf, sumsq = abi.pc_certificate(state["plan"], state["V"], state["idx"], state["x"], state["lam"])
        return dict(mu=mu, mu_inf=torch.tensor(mu_inf, dtype=torch.float32), sumsq=torch.tensor(sumsq, dtype=torch.float32))
    if op == "forward":
        return abi.pc_forward_grid(state["plan"], state["img"])
    if op == "sparse":
        return abi.pc_forward_sparse(state["plan"], state["idx"], state["x"])
    if op == "gram":
        G, b = abi.pc_gram(state["plan"], state["V"], state["idx"])
        return dict(G=G, b=b)
    if op == "apgd":
        x = torch.zeros_like(state["b"])
        x, _, _ = abi.pc_apgd(state["G"], state["b"], state["lam"], 1e-5, 10_000, x)
        return x
    r = abi.pc_solve(state["plan"], state["V"], state["lam"], 0.01)
    img = torch.zeros(state["N"] * state["N"], device=r["x"].device)
    img[r["idx"].long()] = r["x"]          # the reconstructed image
    return dict(img=img.reshape(state["N"], state["N"]), mu=r["mu"])


def work(case):
    N, M, S, op = case["N"], case["M"], case["S"], case["op"]
    # a non-uniform transform: visibilities and their coordinates in single precision, the image once;
    # a transform of the image's size and a 7 x 7 footprint per visibility
    nufft = dict(bytes=20.0 * M + 4.0 * N * N, flops=10.0 * N * N * math.log2(N) + 4.0 * 49 * M)
    if op == "snapshot":
        return dict(bytes=nufft["bytes"] + 12.0 * M, flops=nufft["flops"])
    if op in ("dirty", "forward"):
        return nufft
    if op == "dict":
        return dict(bytes=nufft["bytes"] + 12.0 * N * N, flops=nufft["flops"] + 4.0 * N * N * (9 + 21 + 33))
    if op == "certificate":
        return dict(bytes=nufft["bytes"] + 8.0 * S, flops=nufft["flops"] + 14.0 * M * S)
    if op == "sparse":
        return dict(bytes=20.0 * M + 8.0 * S, flops=14.0 * M * S)
    if op == "gram":
        return dict(bytes=20.0 * M + 4.0 * S * S, flops=2.0 * M * S * (S + 1) + 14.0 * M * S)
    if op == "apgd":
        return dict(bytes=4.0 * S * S + 8.0 * S, flops=100.0 * S * S)   # some fifty products with G
    # a solve: at least the first and the last certificate and the contraction of the sources
    K = case["sources"]
    return dict(bytes=2 * nufft["bytes"], flops=2 * nufft["flops"] + 14.0 * M * K + 2.0 * M * K * K)


# ---------------------------------------------------------------- the same in 64 bits


def _contract(case, uvw, V, idx):
    """Re Phi_S^H Phi_S and Re Phi_S^H V by a direct sum, float64."""
    d, n = _directions(case, idx)
    S = idx.numel()
    G = torch.zeros(S, S, dtype=torch.float64, device="cuda")
    b = torch.zeros(S, dtype=torch.float64, device="cuda")
    step = max(1, 100_000_000 // S)
    for a in range(0, uvw.shape[0], step):
        t = uvw[a:a + step] @ d
        t = (t - torch.round(t)) * (2.0 * math.pi)
        c, s = torch.cos(t), torch.sin(t)
        G += c.T @ c + s.T @ s
        b += V[a:a + step].real.double() @ c - V[a:a + step].imag.double() @ s
    return G / (n[:, None] * n[None, :]), b / n


def _sparse64(case, uvw, idx, x):
    d, n = _directions(case, idx)
    amp = x.double() / n
    out = torch.empty(uvw.shape[0], dtype=torch.complex128, device="cuda")
    step = max(1, 100_000_000 // max(1, idx.numel()))
    for a in range(0, uvw.shape[0], step):
        t = uvw[a:a + step] @ d
        t = (t - torch.round(t)) * (-2.0 * math.pi)
        out[a:a + step] = torch.complex(torch.cos(t) @ amp, torch.sin(t) @ amp)
    return out


_W64 = 14                         # kernel width in cells: about 1e-12 at an oversampling of two


def _es(z):
    return torch.exp(2.3 * _W64 * (torch.sqrt((1.0 - z * z).clamp(min=0.0)) - 1.0))


def _es_transform(t):
    """Fourier transform of the kernel at t cycles per cell."""
    x, w = np.polynomial.legendre.leggauss(80)
    x = torch.tensor(0.5 * (x + 1.0), device="cuda")
    w = torch.tensor(0.5 * w, device="cuda")
    return _W64 * (torch.cos(math.pi * _W64 * t.reshape(-1, 1) * x) @ (w * _es(x))).reshape(t.shape)


class _Nufft64:
    """The dense operators in 64 bits: spreading with a wide kernel over w-planes, torch.fft between."""

    def __init__(self, case, uvw):
        N, fov = case["N"], math.radians(case["fov_deg"])
        self.N, self.G, self.uvw = N, 2 * N, uvw
        dl = fov / N
        ax = (torch.arange(N, device="cuda", dtype=torch.float64) - N / 2)
        l = ax * dl
        r2 = l[:, None] ** 2 + l[None, :] ** 2
        n = torch.sqrt(1.0 - r2)
        s = -r2 / (1.0 + n)
        psi = _es_transform(ax / self.G)
        corr = 1.0 / (n * psi[:, None] * psi[None, :])
        w = uvw[:, 2]
        w_min, w_max = float(w.min()), float(w.max())
        self.cell, self.frac = [], []
        for c in (0, 1):
            g = uvw[:, c] * dl * self.G
            a0 = torch.ceil(g - _W64 / 2)
            self.cell.append(a0.long())
            self.frac.append(g - a0)
        if w_max > w_min:
            s_min = float(s.min())
            s_c = 0.5 * s_min
            dw = 0.5 / -s_min
            w0 = w_min - 0.5 * _W64 * dw
            self.planes = math.ceil((w_max - w_min) / dw) + _W64
            self.x = (w - w0) / dw
            self.tau = torch.polar(torch.ones_like(w), 2.0 * math.pi * (((w - w0) * s_c) % 1.0))
            self.t = dw * (s - s_c)
            corr = corr / _es_transform_fast(self.t)
            self.corr = torch.polar(corr, 2.0 * math.pi * ((w0 * s) % 1.0))
        else:
            self.planes, self.x, self.t = 1, None, None
            self.corr = torch.polar(corr, 2.0 * math.pi * ((w_min * s) % 1.0))
        self.at = (torch.arange(N, device="cuda") - N // 2) % self.G

    def _plane(self, p):
        """Visibilities that meet plane p and their weights in w."""
        if self.x is None:
            return slice(None), None
        z = (self.x - p) * (2.0 / _W64)
        k = (z.abs() < 1.0).nonzero()[:, 0]
        return k, _es(z[k]) * self.tau[k]

    def _taps(self, k):
        a, b = self.cell[0][k], self.cell[1][k]
        fa, fb = self.frac[0][k], self.frac[1][k]
        for j in range(_W64):
            col, wb = (b + j) % self.G, _es((fb - j) * (2.0 / _W64))
            for i in range(_W64):
                yield ((a + i) % self.G) * self.G + col, wb * _es((fa - i) * (2.0 / _W64))

    def adjoint(self, h):
        h = h.to(torch.complex128)
        img = torch.zeros(self.N, self.N, dtype=torch.complex128, device="cuda")
        for p in range(self.planes):
            k, ww = self._plane(p)
            v = h[k] if ww is None else h[k] * ww
            grid = torch.zeros(2, self.G * self.G, dtype=torch.float64, device="cuda")
            for at, wt in self._taps(k):
                grid[0].index_add_(0, at, v.real * wt)
                grid[1].index_add_(0, at, v.imag * wt)
            f = torch.fft.ifft2(torch.complex(grid[0], grid[1]).reshape(self.G, self.G), norm="forward")
            f = f[self.at][:, self.at]
            img += f if ww is None else f * torch.polar(torch.ones_like(self.t), 2.0 * math.pi * ((p * self.t) % 1.0))
        return (img * self.corr).real

    def forward(self, img):
        out = torch.zeros(self.uvw.shape[0], dtype=torch.complex128, device="cuda")
        base = img.double() * self.corr
        for p in range(self.planes):
            k, ww = self._plane(p)
            f = base if ww is None else base * torch.polar(torch.ones_like(self.t), 2.0 * math.pi * ((p * self.t) % 1.0))
            grid = torch.zeros(self.G, self.G, dtype=torch.complex128, device="cuda")
            grid[self.at[:, None], self.at[None, :]] = f
            grid = torch.fft.ifft2(grid, norm="forward").reshape(-1)
            acc = torch.zeros_like(out[k])
            for at, wt in self._taps(k):
                acc += grid[at] * wt
            out[k] += acc if ww is None else acc * ww
        return out.conj().resolve_conj()


def _es_transform_fast(t):
    """The transform over a whole image: a polynomial through Chebyshev points of its narrow range."""
    lo, hi = float(t.min()), float(t.max())
    deg = 40
    x = np.cos(np.pi * (np.arange(deg + 1) + 0.5) / (deg + 1))
    y = _es_transform(torch.tensor(0.5 * (hi + lo) + 0.5 * (hi - lo) * x, device="cuda")).cpu().numpy()
    c = np.polynomial.chebyshev.chebfit(x, y, deg)
    z = (2.0 * t - (hi + lo)) / (hi - lo)
    b1, b2 = torch.zeros_like(z), torch.zeros_like(z)
    for k in range(deg, 0, -1):
        b1, b2 = 2.0 * z * b1 - b2 + float(c[k]), b1
    return z * b1 - b2 + float(c[0])


def exact(case, seed):
    op = case["op"]
    if op in ("apgd", "solve"):
        return None                # iterations that stop early have no value of their own
    uvw = _uvw(case, seed)
    if op == "sparse":
        idx = _pixels(case, seed, 5, case["S"])
        x = torch.exp(torch.randn(idx.numel(), generator=_generator(seed, 6), device="cuda"))
        return _sparse64(case, uvw, idx, x)
    if op == "forward":
        return _Nufft64(case, uvw).forward(_dense_image(case, seed))
    V, idx, flux = _visibilities(case, seed, uvw)
    if op == "gram":
        G, b = _contract(case, uvw, V, _atoms(case, seed))
        return dict(G=G, b=b)
    if op == "certificate":
        at, x = _support(case, seed, idx, flux)
        r = V.to(torch.complex128) - _sparse64(case, uvw, at, x)
        mu = _Nufft64(case, uvw).adjoint(r) / (0.1 * case["M"] * float(flux.max()))
        return dict(mu=mu, mu_inf=mu.abs().max(), sumsq=(r.real ** 2 + r.imag ** 2).sum())
    img = _Nufft64(case, uvw).adjoint(V)
    if op != "dict":
        return img
    out, d = [], _dictionary()
    for i in range(d.n_scales):
        r = int(math.floor(2.0 * d.sigma[i]))
        k = torch.ones(1, device="cuda", dtype=torch.float64)
        if r:
            a = torch.arange(-r, r + 1, device="cuda", dtype=torch.float64)
            k = torch.exp(-(a / d.sigma[i]) ** 2)
            k = k / k.sum()
        f = torch.nn.functional.conv2d(img[None, None], k.reshape(1, 1, -1, 1), padding=(r, 0))
        f = torch.nn.functional.conv2d(f, k.reshape(1, 1, 1, -1), padding=(0, r))
        out.append(d.gamma[i] * f[0, 0])
    return torch.stack(out)
