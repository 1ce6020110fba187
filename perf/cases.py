"""Reconstruction workloads of the library, as a user's program calls them through the Python binding.

A pass starts where new data arrive: the plan (sizes, prior, weights) is in hand, the measurements y
are on the GPU, and the pass sets them, iterates and reads the results back.  In cases with
``"psfs": "new"`` the PSFs arrive with the data, so the factor is formed inside the pass too;
otherwise the plan already holds it, as in a camera or spectrometer whose optics stay fixed.

``exact`` runs the same iterations (Dogan & Oktem, arXiv 2006.08303, Alg. 1 and Alg. 2) in 64 bits
with plain torch.
"""
from __future__ import annotations

import math
import random

import torch

from paper_2006_08303_gb300 import api

DEV = "cuda"

# prior -> (lambda, rho, beta): the weights of the repository's workloads
WEIGHTS = {"tv": (1e-2, 1.0, 1.0), "tv_iso": (1e-2, 1.0, 1.0), "dct8": (1e-3, 1e-2, 1.0), "l1": (1e-3, 1e-2, 1.0),
           "wdct": (1e-3, 1e-2, 1.0), "convdict": (0.15, 8.0, 4.0)}
SNR_DB = {"convdict": 25.0}
SIGMA = 10.0  # filter penalty of the online dictionary update


def listed():
    return [
        # the smallest image of the configurations: launches and latency are all there is
        {"name": "tv_64x64x3", "kind": "analysis", "prior": "tv", "N": 64, "K": 3, "M": 3, "iters": 50,
         "dtype": "f32", "psfs": "kept"},
        # the benchmark workload: PSFs and measurements arrive together, block-DCT prior
        {"name": "dct_512x512x10_full", "kind": "analysis", "prior": "dct8", "N": 512, "K": 10, "M": 10, "iters": 100,
         "dtype": "f32", "psfs": "new"},
        # a spectral image whose iteration no longer fits the L2 cache, next frame of a fixed instrument
        {"name": "dct_1024x1024x10", "kind": "analysis", "prior": "dct8", "N": 1024, "K": 10, "M": 10, "iters": 40,
         "dtype": "f32", "psfs": "kept"},
        # TV to a tolerance with the penalty adapted from a poor start, as the served requests run it
        {"name": "tv_512x512x5_adaptive", "kind": "adaptive", "prior": "tv", "N": 512, "K": 5, "M": 5, "iters": 200,
         "tol": 3e-4, "rho0": 8.0, "dtype": "f32", "psfs": "kept"},
        # multiframe data: more measurements than channels, isotropic TV
        {"name": "tv_iso_256x256x3_k4", "kind": "analysis", "prior": "tv_iso", "N": 256, "K": 4, "M": 3, "iters": 100,
         "dtype": "f32", "psfs": "kept"},
        # the largest image side
        {"name": "tv_2048x2048x3", "kind": "analysis", "prior": "tv", "N": 2048, "K": 3, "M": 3, "iters": 20,
         "dtype": "f32", "psfs": "kept"},
        # Kronecker wavelet x channel-DCT prior
        {"name": "wdct_512x512x10", "kind": "analysis", "prior": "wdct", "N": 512, "K": 10, "M": 10, "iters": 40,
         "dtype": "f32", "psfs": "kept"},
        # convolutional dictionary, fixed filters
        {"name": "convdict_256x256x5_l32", "kind": "convdict", "prior": "convdict", "N": 256, "K": 5, "M": 5, "L": 32,
         "P": 11, "mu": 0.0, "iters": 60, "dtype": "f32", "psfs": "kept"},
        # the same while the filters are learnt online: the image is what is read back
        {"name": "dictlearn_256x256x5_l32", "kind": "dictlearn", "prior": "convdict", "N": 256, "K": 5, "M": 5,
         "L": 32, "P": 11, "iters": 15, "dtype": "f32", "psfs": "kept"},
        # 3D dictionary over a spectral cube
        {"name": "convdict3d_256x256x16_l6", "kind": "convdict3d", "prior": "convdict", "N": 256, "K": 16, "M": 16,
         "L": 6, "Q": 5, "P": 11, "iters": 30, "dtype": "f32", "psfs": "kept"},
        # double precision (complex128 plan)
        {"name": "dct_256x256x5_f64", "kind": "analysis", "prior": "dct8", "N": 256, "K": 5, "M": 5, "iters": 40,
         "dtype": "f64", "psfs": "new"},
        # many independent uneven instances iterated together
        {"name": "batch_16_mixed", "kind": "batch", "prior": "tv", "members": 16, "mix": 1, "iters": 60,
         "dtype": "f32", "psfs": "kept"},
    ]


def _batch_members(case):
    """(N, M) of every instance of a batch: N over {128, 256, 512}, M = K over {3, 5, 10}."""
    r = random.Random(case["mix"])
    return [(r.choice((128, 256, 512)), r.choice((3, 5, 10))) for _ in range(case["members"])]


def draw(rng):
    most = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(("analysis",) * 6 + ("adaptive", "convdict", "dictlearn", "convdict3d", "batch"))
        iters = int(round(math.exp(rng.uniform(math.log(10), math.log(100)))))
        c = {"kind": kind, "iters": iters, "dtype": "f32", "psfs": "kept"}
        if kind == "analysis":
            c["prior"] = rng.choice(("tv", "tv_iso", "dct8", "l1", "wdct"))
            c["N"] = 2 ** rng.randint(6, 11)
            c["M"] = rng.randint(1, 16)
            c["K"] = c["M"] if rng.random() < 0.6 else rng.randint(1, 16)
            c["dtype"] = "f64" if rng.random() < 0.15 else "f32"
            c["psfs"] = rng.choice(("kept", "kept", "new"))
            if c["prior"] in ("dct8", "l1", "wdct"):
                c["iters"] = min(iters, 60)
            if c["N"] == 2048:
                c["iters"] = min(iters, 20)
        elif kind == "adaptive":
            c.update(prior="tv", N=2 ** rng.randint(7, 9), M=rng.randint(1, 10), tol=3e-4, rho0=8.0,
                     iters=rng.randint(6, 20) * 10)
            c["K"] = c["M"]
        elif kind == "convdict":
            c.update(prior="convdict", N=2 ** rng.randint(6, 9), M=rng.randint(1, 10), L=rng.randint(1, 32),
                     P=rng.randint(1, 8) * 2 + 1, mu=rng.choice((0.0, 0.0, 0.5)))
            c["K"] = c["M"]
        elif kind == "dictlearn":
            c.update(prior="convdict", N=2 ** rng.randint(6, 9), M=rng.randint(1, 8), L=rng.randint(1, 32),
                     P=rng.randint(1, 8) * 2 + 1, iters=rng.randint(5, 15))
            c["K"] = c["M"]
        elif kind == "convdict3d":
            c.update(prior="convdict", N=2 ** rng.randint(6, 8), M=rng.randint(2, 16), L=rng.randint(1, 8),
                     P=rng.randint(1, 7) * 2 + 1)
            c["K"] = c["M"]
            c["Q"] = rng.randint(1, min(5, c["M"]))
        else:
            c.update(prior="tv", members=rng.randint(2, 24), mix=rng.randint(0, 1 << 20))
        if _cost(c) <= most:
            return c


# ---------------------------------------------------------------------------------------------
# inputs: seeded images, PSFs and measurements with the structure of the repository's generators
# ---------------------------------------------------------------------------------------------
def _gaussian(N, s):
    d = torch.arange(N, device=DEV, dtype=torch.float64)
    d = torch.minimum(d, N - d)
    e = torch.exp(-0.5 * d * d / (s * s))
    h = e[:, None] * e[None, :]
    return h / h.sum()


def _psfs(N, K, M, prior, r):
    """Unit-sum PSFs [K][M][N][N] whose width grows with |k - m|: Gaussians, or disks convolved with a
    1 px Gaussian for the spectral priors; the instrument's defocus varies a little with the seed."""
    f = r.uniform(0.95, 1.05)
    bank = {}
    for a in {abs(k - m) for k in range(K) for m in range(M)}:
        if prior in ("tv", "tv_iso", "convdict"):
            bank[a] = _gaussian(N, f * (0.5 + 1.5 * a))
        else:
            rad = f * 12.0 * a / max(max(K, M) - 1, 1)
            d = torch.arange(N, device=DEV, dtype=torch.float64)
            d = torch.minimum(d, N - d)
            disk = ((d[:, None] ** 2 + d[None, :] ** 2).sqrt() <= rad + 1e-12).double()
            h = torch.fft.irfft2(torch.fft.rfft2(disk / disk.sum()) * torch.fft.rfft2(_gaussian(N, 1.0)), s=(N, N))
            h = h.clamp_min(0.0)
            bank[a] = h / h.sum()
    return torch.stack([torch.stack([bank[abs(k - m)] for m in range(M)]) for k in range(K)])


def _image(N, M, prior, r, gen):
    """Additive rectangles (TV), or piecewise-constant cells times smooth spectra (spectral priors)."""
    if prior in ("tv", "tv_iso"):
        x = torch.zeros(M, N, N, device=DEV, dtype=torch.float64)
        n = torch.arange(N, device=DEV)
        for m in range(M):
            for _ in range(8):
                rows = (n - r.randrange(N)) % N < r.randint(4, max(4, N // 4))
                cols = (n - r.randrange(N)) % N < r.randint(4, max(4, N // 4))
                x[m] += r.random() * (rows[:, None] & cols[None, :])
        return x
    n = torch.arange(N, device=DEV, dtype=torch.float64)
    dist = []
    for _ in range(16):
        a, b = (n - r.uniform(0, N)).abs(), (n - r.uniform(0, N)).abs()
        dist.append(torch.minimum(a, N - a)[:, None] ** 2 + torch.minimum(b, N - b)[None, :] ** 2)
    label = torch.stack(dist).argmin(0)
    ch = torch.arange(M, device=DEV, dtype=torch.float64)
    spec = torch.zeros(16, M, device=DEV, dtype=torch.float64)
    for c in range(16):
        for _ in range(3):
            spec[c] += r.uniform(0.2, 1.0) * torch.exp(
                -0.5 * ((ch - r.uniform(0.0, max(M - 1, 0))) / r.uniform(1.0, max(M / 2.0, 1.0))) ** 2)
    return spec[label].permute(2, 0, 1).contiguous()


def _gabor(L, P, r):
    """Zero-mean unit-norm Gabor filters [L][P][P]."""
    n = torch.arange(P, device=DEV, dtype=torch.float64) - P // 2
    v, u = n[:, None], n[None, :]
    out = []
    for _ in range(L):
        th, sg, ph = r.uniform(0, math.pi), r.uniform(1.5, 3.5), r.uniform(0, 2 * math.pi)
        d = torch.exp(-(u * u + v * v) / (2 * sg * sg)) * torch.cos(
            2 * math.pi * (u * math.cos(th) + v * math.sin(th)) / (2.5 * sg) + ph)
        d = d - d.mean()
        out.append(d / d.norm())
    return torch.stack(out)


def _embed(d, N):
    """P x P filters on the N x N torus, centre at (0, 0)."""
    P = d.shape[-1]
    out = torch.zeros(*d.shape[:-2], N, N, device=DEV, dtype=torch.float64)
    idx = (torch.arange(P, device=DEV) - P // 2) % N
    out[..., idx[:, None], idx[None, :]] = d.double()
    return out


def _embed3(d, N, S):
    """Q x P x P filters on the S x N x N torus, centre at (0, 0, 0)."""
    L, Q = d.shape[:2]
    out = torch.zeros(L, S, N, N, device=DEV, dtype=torch.float64)
    out[:, (torch.arange(Q, device=DEV) - Q // 2) % S] = _embed(d, N)
    return out


def _codes(L, M, N, gen):
    """1% Bernoulli-Gaussian code maps [L][M][N][N]."""
    on = torch.rand(L, M, N, N, device=DEV, generator=gen) < 0.01
    return on * torch.randn(L, M, N, N, device=DEV, generator=gen, dtype=torch.float64)


def _inputs(case, seed, N, K, M):
    """PSFs h [K][M][N][N], measurements y [K][N][N] and (dictionary priors) filters, in the plan's type."""
    r = random.Random(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    prior, t = case["prior"], torch.float64 if case["dtype"] == "f64" else torch.float32
    d = None
    if case["kind"] in ("convdict", "dictlearn"):
        d = _gabor(case["L"], case["P"], r)
        Z = torch.fft.rfft2(_codes(case["L"], M, N, gen))
        x = torch.fft.irfft2(torch.einsum("lab,lmab->mab", torch.fft.rfft2(_embed(d, N)), Z), s=(N, N))
        if case["kind"] == "dictlearn":  # learning starts from other filters than the scene's
            d = _gabor(case["L"], case["P"], r)
    elif case["kind"] == "convdict3d":
        L, Q = case["L"], case["Q"]
        prof = torch.exp(-0.5 * ((torch.arange(Q, device=DEV, dtype=torch.float64) - Q // 2) / 1.0) ** 2)
        d = prof[None, :, None, None] * _gabor(L, case["P"], r)[:, None]
        d = d / d.flatten(1).norm(dim=1)[:, None, None, None]
        X = (torch.fft.rfftn(_embed3(d, N, M), dim=(1, 2, 3)) * torch.fft.rfftn(_codes(L, M, N, gen), dim=(1, 2, 3))).sum(0)
        x = torch.fft.irfftn(X, s=(M, N, N))
    else:
        x = _image(N, M, prior, r, gen)
    h = _psfs(N, K, M, prior, r)
    X, clean = torch.fft.rfft2(x), []
    for k in range(K):
        clean.append(torch.fft.irfft2((torch.fft.rfft2(h[k]) * X).sum(0), s=(N, N)))
    clean = torch.stack(clean)
    s = (clean.square().mean() / 10.0 ** (SNR_DB.get(prior, 30.0) / 10.0)).sqrt()
    y = clean + s * torch.randn(K, N, N, device=DEV, generator=gen, dtype=torch.float64)
    return h.to(t).contiguous(), y.to(t).contiguous(), None if d is None else d.to(t).contiguous()


def _plan(case, N, K, M, h, d):
    p = api.Plan(N, K, M, case["dtype"])
    lam, rho, beta = WEIGHTS[case["prior"]]
    p.set_prior(case["prior"], lam, case.get("rho0", rho), beta)
    if case["kind"] == "convdict3d":
        p.set_dictionary_3d(d)
    elif d is not None:
        p.set_dictionary(d)
        if case.get("mu", 0.0):
            p.set_code_gradient_weight(case["mu"])
    if case["kind"] == "adaptive":
        p.set_rho_adaptation(2.0, 10.0)
    if case["psfs"] == "kept":
        p.set_psfs(h)
    return p


# ---------------------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------------------
def prepare(case, seed):
    if case["kind"] == "batch":
        plans, ys = [], []
        for i, (N, M) in enumerate(_batch_members(case)):
            h, y, _ = _inputs(case, seed * 1009 + i, N, M, M)
            plans.append(_plan(case, N, M, M, h, None))
            ys.append(y)
        return {"case": case, "plans": plans, "y": ys, "batch": api.Batch(plans)}
    N, K, M = case["N"], case["K"], case["M"]
    h, y, d = _inputs(case, seed, N, K, M)
    return {"case": case, "plan": _plan(case, N, K, M, h, d), "h": h if case["psfs"] == "new" else None, "y": y, "d": d}


def run(state):
    case = state["case"]
    n = case["iters"]
    if case["kind"] == "batch":
        for p, y in zip(state["plans"], state["y"]):
            p.set_measurements(y)
        state["batch"].iterate(n)
        return [p.get_x() for p in state["plans"]]
    p = state["plan"]
    if case["kind"] == "adaptive":  # the next frame starts from the first penalty again
        lam, _, beta = WEIGHTS[case["prior"]]
        p.set_prior(case["prior"], lam, case["rho0"], beta)
    if case["kind"] == "dictlearn":  # every frame learns from the same first filters
        p.set_dictionary(state["d"])
        p.set_dictionary_learning(SIGMA)
    if state["h"] is not None:
        p.set_psfs(state["h"])
    p.set_measurements(state["y"])
    done = p.iterate(n, case.get("tol", 0.0))
    out = {"x": p.get_x()}
    if case["kind"] == "adaptive":
        out["iterations"] = done
        out["rho"] = p.rho
    elif case["kind"] in ("convdict", "convdict3d"):
        out["z"] = p.get_coefficients()
    return out


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _one(kind, prior, N, K, M, iters, dtype, psfs, L=0):
    """(bytes, flops) of one instance.  An iteration reads the factor and the data term, reads and
    writes the state (the scaled dual), and exchanges the spectra of the maps between the row and the
    column half of the 2D transforms, both ways; nothing is counted twice."""
    r = 8 if dtype == "f64" else 4
    half, pix, tri = N * (N // 2 + 1), N * N, M * (M + 1) // 2
    lg = math.log2(N)
    S = M * L if L else M
    nc = 2 if prior in ("tv", "tv_iso") else 1
    it_b = (tri + M + 4 * S) * half * 2 * r + 2 * nc * S * pix * r
    it_f = S * 2 * 5.0 * pix * lg + 8.0 * M * M * half + 8.0 * nc * S * pix
    if prior == "dct8":
        it_f += 2 * 2 * 36.0 / 8 * S * pix
    if prior == "wdct":
        it_f += 2 * (64.0 * 4 / 3 + 2 * M) * S * pix
    if L:  # theta, p in and out, x; the per-bin solves
        th = L * M if kind == "convdict3d" else L
        it_b += (th + 3 * M) * half * 2 * r
        it_f += 32.0 * S * half + (16.0 * M * S * half if kind == "convdict3d" else 0.0)
    if kind == "dictlearn":  # codes once more, w, theta and the dual's spectrum
        it_b += (S + 4 * L) * half * 2 * r
        it_f += (8.0 * M * M + 32.0 * M) * L * half
    b = iters * it_b + K * pix * r + M * pix * r + M * half * 2 * r
    f = iters * it_f + K * 5.0 * pix * lg + 8.0 * (K * M + M * M) * half
    if psfs == "new":
        b += K * M * pix * r + tri * half * 2 * r
        f += K * M * 5.0 * pix * lg + (4.0 * K * M * M + 8.0 * M ** 3) * half
    return b, f


def work(case):
    if case["kind"] == "batch":
        sizes = [(N, M, M) for N, M in _batch_members(case)]
    else:
        sizes = [(case["N"], case["K"], case["M"])]
    b = f = 0.0
    for N, K, M in sizes:
        x, y = _one(case["kind"], case["prior"], N, K, M, case["iters"], case["dtype"], case["psfs"], case.get("L", 0))
        b, f = b + x, f + y
    return {"bytes": b, "flops": f}


def _cost(case):
    """What a drawn case may cost at most: its bytes, more for FP64 arithmetic and for small images."""
    w = work(case)
    n = case["members"] if case["kind"] == "batch" else 1
    per_iter = {"wdct": 100e3, "convdict": 50e3}.get(case["prior"], 20e3) * 100
    return (w["bytes"] + n * case["iters"] * per_iter) * (4.0 if case["dtype"] == "f64" else 1.0)


# ---------------------------------------------------------------------------------------------
# the same iterations in 64 bits
# ---------------------------------------------------------------------------------------------
def _soft(v, tau):
    return torch.sign(v) * (v.abs() - tau).clamp_min(0.0)


def _dct_matrix(n):
    k = torch.arange(n, device=DEV, dtype=torch.float64)[:, None]
    m = torch.arange(n, device=DEV, dtype=torch.float64)[None, :]
    c = torch.cos(math.pi * (2 * m + 1) * k / (2 * n)) * math.sqrt(2.0 / n)
    c[0] = math.sqrt(1.0 / n)
    return c


class _TV:
    """[D_h; D_v]: circular forward differences; x [M][N][N] -> [M][2][N][N]."""

    def fwd(self, x):
        return torch.stack([x.roll(-1, 2) - x, x.roll(-1, 1) - x], 1)

    def adj(self, a):
        h, v = a[:, 0], a[:, 1]
        return h.roll(1, 2) - h + v.roll(1, 1) - v


class _DCT:
    """Orthonormal DCT-II of 8 x 8 blocks."""

    def __init__(self):
        self.c = _dct_matrix(8)

    def _both(self, x, c):
        M, N = x.shape[0], x.shape[-1]
        b = x.reshape(M, N // 8, 8, N // 8, 8)
        return torch.einsum("ki,mainj,lj->maknl", c, b, c).reshape(M, N, N)

    def fwd(self, x):
        return self._both(x, self.c)[:, None]

    def adj(self, a):
        return self._both(a[:, 0], self.c.T)


class _Id:
    def fwd(self, x):
        return x[:, None]

    def adj(self, a):
        return a[:, 0]


class _Wave:
    """Periodic 2D Symmlet-8 levels down to 16 x 16 (Mallat layout), then the DCT-II along the channels."""

    def __init__(self, N, M):
        # from the filter's definition: 8 vanishing moments, |m0|^2 = cos^16 P(sin^2), one root of every
        # reciprocal pair, the choice whose phase is closest to linear, the mirror image with the earlier energy
        import numpy as np
        p = 8
        a = [math.comb(p - 1 + k, k) for k in range(p)]
        ys = np.roots(a[::-1])
        groups, used = [], [False] * len(ys)
        for i, y in enumerate(ys):
            if used[i]:
                continue
            used[i] = True
            w = 1 - 2 * y
            z = w + np.sqrt(w * w - 1 + 0j)
            z = z if abs(z) < 1 else 1 / z
            if abs(y.imag) <= 1e-9 * max(1, abs(y)):
                groups.append([z.real])
            else:
                j = min((q for q in range(len(ys)) if not used[q]), key=lambda q: abs(ys[q] - np.conj(y)))
                used[j] = True
                groups.append([z, np.conj(z)])
        om, best = np.linspace(0, np.pi, 513), []
        for pick in range(1 << len(groups)):
            roots = [1 / z if (pick >> g) & 1 else z for g, zs in enumerate(groups) for z in zs]
            q = np.array([1.0 + 0j])
            for z in roots:
                q = np.convolve(q, [1.0, -z])
            for _ in range(p):
                q = np.convolve(q, [1.0, 1.0])
            h = q.real * math.sqrt(2.0) / q.real.sum()
            ph = np.unwrap(np.angle(np.prod([1 - z * np.exp(-1j * om) for z in roots], axis=0)))
            dev = float(np.sum((ph - np.polyval(np.polyfit(om, ph, 1), om)) ** 2))
            best.append((dev, float(np.sum(np.arange(16) * h * h)), h))
        low = min(b[0] for b in best)
        h = min((b for b in best if b[0] - low <= 1e-6 * max(1.0, low)), key=lambda b: b[1])[2]
        g = np.array([(-1) ** k * h[15 - k] for k in range(16)])
        self.levels, n = [], N
        while n > 16:
            W = torch.zeros(n, n, dtype=torch.float64)
            for i in range(n // 2):
                for k in range(16):
                    W[i, (2 * i + k) % n] += h[k]
                    W[n // 2 + i, (2 * i + k) % n] += g[k]
            self.levels.append(W.to(DEV))
            n //= 2
        self.c = _dct_matrix(M)

    def fwd(self, x):
        a = x.clone()
        for W in self.levels:
            n = W.shape[0]
            a[:, :n, :n] = W @ a[:, :n, :n] @ W.T
        return torch.einsum("km,mab->kab", self.c, a)[:, None]

    def adj(self, t):
        a = torch.einsum("km,kab->mab", self.c, t[:, 0])
        for W in reversed(self.levels):
            n = W.shape[0]
            a[:, :n, :n] = W.T @ a[:, :n, :n] @ W
        return a


def _operator(prior, N, M):
    return _TV() if prior in ("tv", "tv_iso") else _DCT() if prior == "dct8" else _Id() if prior == "l1" else _Wave(N, M)


def _grad_eig(N):
    s = 4 * torch.sin(math.pi * torch.arange(N, device=DEV, dtype=torch.float64) / N) ** 2
    return s[:, None] + s[None, : N // 2 + 1]


def _spectra(h, y):
    """Lambda [N][H][K][M] and F y [N][H][K]."""
    return torch.fft.rfft2(h.double()).permute(2, 3, 0, 1), torch.fft.rfft2(y.double()).permute(1, 2, 0)


def _inverse(Lam, diag, beta):
    """(diag I + beta Lambda^H Lambda)^-1 per bin, the min-norm inverse where diag is 0."""
    M = Lam.shape[-1]
    eye = torch.eye(M, device=DEV, dtype=torch.complex128)
    Psi = diag[..., None, None] * eye + beta * (Lam.conj().transpose(-1, -2) @ Lam)
    sing = diag == 0
    fix = Psi[sing]
    Psi[sing] = eye
    inv = torch.linalg.inv(Psi)
    if fix.shape[0]:
        inv[sing] = torch.linalg.pinv(fix, hermitian=True, rtol=1e-10)
    return inv


def _to_image(X, N):
    return torch.fft.irfft2(X.permute(2, 0, 1), s=(N, N))


def _exact_analysis(case, h, y, N, K, M):
    prior = case["prior"]
    lam, rho, beta = WEIGHTS[prior]
    rho = case.get("rho0", rho)
    T = _operator(prior, N, M)
    Lam, Y = _spectra(h, y)
    g = _grad_eig(N) if prior in ("tv", "tv_iso") else torch.ones(N, N // 2 + 1, device=DEV, dtype=torch.float64)
    b = beta * (Lam.conj().transpose(-1, -2) @ Y[..., None])
    P = _inverse(Lam, rho * g, beta)
    nc = 2 if prior in ("tv", "tv_iso") else 1
    t = torch.zeros(M, nc, N, N, device=DEV, dtype=torch.float64)
    u = torch.zeros_like(t)
    adaptive, tol, done = case["kind"] == "adaptive", case.get("tol", 0.0), 0
    for it in range(case["iters"]):
        Q = torch.fft.rfft2(T.adj(t - u)).permute(1, 2, 0)[..., None]
        x = _to_image((P @ (b + rho * Q))[..., 0], N)
        w = T.fwd(x)
        v = w + u
        if prior == "tv_iso":
            nrm = v.square().sum(1, keepdim=True).sqrt()
            tn = v * torch.where(nrm > lam / rho, 1 - (lam / rho) / nrm, torch.zeros_like(nrm))
        else:
            tn = _soft(v, lam / rho)
        u = v - tn
        done = it + 1
        if adaptive and done % 10 == 0:
            pr, du = float((w - tn).norm()), rho * float((tn - t).norm())
            if tol > 0 and done < case["iters"] and pr < tol * max(float(w.norm()), float(tn.norm())) and du < tol * rho * float(u.norm()):
                break
            new = rho * 2 if pr > 10 * du else rho / 2 if du > 10 * pr else rho
            if new != rho:
                u, rho = u * (rho / new), new
                P = _inverse(Lam, rho * g, beta)
        t = tn
    if adaptive:
        return {"x": x, "iterations": done, "rho": rho}
    return x if case["kind"] == "batch" else {"x": x}


def _project(v, P):
    """Filters on the torus cut to their P x P support and scaled to unit norm."""
    N = v.shape[-1]
    idx = (torch.arange(P, device=DEV) - P // 2) % N
    c = v[:, idx[:, None], idx[None, :]]
    return c / c.flatten(1).norm(dim=1)[:, None, None]


def _exact_dictionary(case, h, y, d, N, K, M):
    lam, rho, beta = WEIGHTS["convdict"]
    Lam, Y = _spectra(h, y)
    P = _inverse(Lam, torch.ones(N, N // 2 + 1, device=DEV, dtype=torch.float64), beta)
    b = beta * (Lam.conj().transpose(-1, -2) @ Y[..., None])
    L, three = case["L"], case["kind"] == "convdict3d"
    th = torch.fft.fft(torch.fft.rfft2(_embed3(d, N, M)), dim=1) if three else torch.fft.rfft2(_embed(d, N))[:, None]
    rn = rho + case.get("mu", 0.0) * _grad_eig(N)
    fwd = (lambda a: torch.fft.fft(torch.fft.rfft2(a), dim=1)) if three else torch.fft.rfft2
    z = torch.zeros(L, M, N, N, device=DEV, dtype=torch.float64)
    t, u = torch.zeros_like(z), torch.zeros_like(z)
    learn = case["kind"] == "dictlearn"
    g, e = _embed(d, N) if learn else None, 0.0
    for _ in range(case["iters"]):
        if learn:
            th = torch.fft.rfft2(g)[:, None]
        p = (th * fwd(z)).sum(0)
        p = torch.fft.ifft(p, dim=0) if three else p
        X = (P @ (b + p.permute(1, 2, 0)[..., None]))[..., 0]
        x = _to_image(X, N)
        X = X.permute(2, 0, 1)
        c = th.conj() * (torch.fft.fft(X, dim=0) if three else X) + rho * fwd(t - u)
        v = (c - th.conj() * (th * c).sum(0) / (rn + th.abs().square().sum(0))) / rn
        v = torch.fft.ifft(v, dim=1) if three else v
        z = torch.fft.irfft2(v, s=(N, N))
        t = _soft(z + u, lam / rho)
        u = u + z - t
        if learn:
            Zh, Xh = torch.fft.rfft2(z).permute(2, 3, 1, 0), torch.fft.rfft2(x).permute(1, 2, 0)  # [N][H][M][L], [N][H][M]
            r = (Zh.conj() * Xh[..., None]).sum(-2) + SIGMA * torch.fft.rfft2(g - e).permute(1, 2, 0)
            S = SIGMA * torch.eye(M, device=DEV, dtype=torch.complex128) + Zh @ Zh.conj().transpose(-1, -2)
            al = torch.linalg.solve(S, Zh @ r[..., None])
            D = (r - (Zh.conj().transpose(-1, -2) @ al)[..., 0]) / SIGMA
            s = _to_image(D, N) + e
            g = _embed(_project(s, case["P"]), N)
            e = s - g
    return {"x": x} if learn else {"x": x, "z": z.transpose(0, 1).contiguous()}


def exact(case, seed):
    with torch.no_grad():
        if case["kind"] == "batch":
            out = []
            for i, (N, M) in enumerate(_batch_members(case)):
                h, y, _ = _inputs(case, seed * 1009 + i, N, M, M)
                out.append(_exact_analysis(case, h, y, N, M, M))
            return out
        N, K, M = case["N"], case["K"], case["M"]
        h, y, d = _inputs(case, seed, N, K, M)
        if d is not None:
            return _exact_dictionary(case, h, y, d, N, K, M)
        return _exact_analysis(case, h, y, N, K, M)
