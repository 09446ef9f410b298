"""The work a user of this library has it do, as measurable cases.

Every case goes through the public binding: the operator pairs Phi / Phi^H and
Psi^H / Psi, the normal operator of the CG update in both its forms, whole
SARA and TV solves on device data, the batched solver and the end-to-end call
on host buffers.  Inputs are made from the seed alone: a sky of Gaussian blobs
and point sources, a Gaussian variable-density uv coverage with its (0, 0)
cell suppressed, and visibilities from the sky's analytic Fourier transform
plus noise of 30 dB input SNR -- like a measurement, they owe nothing to the
operator under test.  ``exact`` restates each output in 64 bits with plain
torch / numpy.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1406_0359_gb300 import binding

J = 8  # Kaiser-Bessel support in grid cells, oversampling 2
ALL_BASES = 0x1FF


# ------------------------------------------------------------------ the cases
def listed() -> list[dict]:
    return [
        # the smallest imaging configuration (64^2 sky, 4096 uv points): launches and latency are all of it
        dict(name="phi_64", op="phi", n=64, M=4096, prec="fp32"),
        # prediction of all visibilities from a model image at the benchmark's size
        dict(name="phi_1024", op="phi", n=1024, M=4194304, prec="fp32"),
        # the dirty image of the same data set
        dict(name="phi_adj_1024", op="phi_adj", n=1024, M=4194304, prec="fp32"),
        # the dirty image at the paper's size in double precision, the library's check on its own rounding
        dict(name="phi_adj_256_f64", op="phi_adj", n=256, M=131072, prec="fp64"),
        # the CG operator of every solve up to 1024^2: Phi^H Phi as a precomputed convolution
        dict(name="gram_1024", op="gram", mode=1, n=1024, M=4194304, prec="fp32"),
        # the CG operator of the largest images served (2048^2): Phi^H Phi through the grid; a ragged number of points
        dict(name="gram_2048_nufft", op="gram", mode=0, n=2048, M=1500007, prec="fp32"),
        # the SARA analysis and synthesis of a large image
        dict(name="sara_fwd_1024", op="sara_fwd", n=1024, levels=4, mask=ALL_BASES, prec="fp32"),
        dict(name="sara_adj_1024", op="sara_adj", n=1024, levels=4, mask=ALL_BASES, prec="fp32"),
        # the benchmark's solve: 20 SDMM iterations at 1024^2 / 4,194,304 points
        dict(name="solve_1024", op="solve", n=1024, M=4194304, levels=4, prior="l1", mask=ALL_BASES, blocks=1,
             t_max=20, n_reweight=0, prec="fp32"),
        # the comparison prior (total variation) at a middling size, an odd number of points
        dict(name="solve_512_tv", op="solve", n=512, M=393217, levels=4, prior="tv", mask=ALL_BASES, blocks=1,
             t_max=20, n_reweight=0, prec="fp32"),
        # many independent fields or channels at once
        dict(name="batch_16", op="batch", count=16, pick=40, levels=3, t_max=10, prec="fp32"),
        # uv and y in host memory to an image in host memory at the paper's size, with one reweighting
        dict(name="image_256_host", op="image", n=256, M=131072, levels=4, t_max=30, n_reweight=1, prec="fp32"),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng: random.Random) -> dict:
    op = rng.choice(["phi", "phi", "phi_adj", "phi_adj", "gram", "gram", "sara_fwd", "sara_adj", "solve", "solve",
                     "batch", "image"])
    prec = "fp64" if rng.random() < 0.2 else "fp32"
    if op in ("phi", "phi_adj"):
        n = 1 << rng.randint(5, 11)
        return dict(op=op, n=n, M=_log_int(rng, 64, 4194304 if prec == "fp32" else 300000), prec=prec)
    if op == "gram":
        mode = rng.choice([0, 1, 1])
        n = 1 << (rng.randint(6, 10) if mode else rng.randint(5, 11))
        if prec == "fp64":
            n = min(n, 512)
        return dict(op=op, mode=mode, n=n, M=_log_int(rng, 1000, 1500000 if prec == "fp32" else 200000), prec=prec)
    if op in ("sara_fwd", "sara_adj"):
        n = 1 << rng.randint(5, 10)
        mask = rng.choice([ALL_BASES, ALL_BASES, ALL_BASES, 1 << 8, rng.randint(1, ALL_BASES)])
        return dict(op=op, n=n, levels=rng.randint(1, min(6, n.bit_length() - 2)), mask=mask, prec=prec)
    if op == "solve":
        n = 1 << rng.randint(6, 9)
        return dict(op=op, n=n, M=_log_int(rng, n * n // 4, 3 * n * n if prec == "fp32" else n * n), levels=rng.randint(2, 4),
                    prior=rng.choice(["l1", "l1", "tv"]), mask=rng.choice([ALL_BASES, ALL_BASES, 1 << 8]),
                    blocks=rng.choice([1, 1, 3]), t_max=rng.randint(3, 12), n_reweight=rng.choice([0, 1]), prec=prec)
    if op == "batch":
        return dict(op=op, count=rng.randint(2, 16), pick=rng.randint(0, 1 << 20), levels=3, t_max=rng.randint(3, 10),
                    prec="fp32")
    n = 1 << rng.randint(6, 9)
    return dict(op=op, n=n, M=_log_int(rng, n * n // 4, 3 * n * n), levels=3, t_max=rng.randint(5, 20),
                n_reweight=rng.choice([0, 1]), prec="fp32")


def _members(case: dict) -> list[dict]:
    """The instances of a batch: image sides 128..512, M in [0.5 N, 3 N]."""
    r = random.Random(case["pick"])
    out = []
    for _ in range(case["count"]):
        n = r.choice([128, 256, 512])
        out.append(dict(n=n, M=int(r.uniform(0.5, 3.0) * n * n)))
    return out


# ------------------------------------------------------------------ inputs
def _device() -> torch.device:
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _generator(seed: int) -> torch.Generator:
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _uniform(g, lo, hi, size):
    return lo + (hi - lo) * torch.rand(size, generator=g, device=g.device, dtype=torch.float64)


def _coverage(g, M: int, n: int) -> torch.Tensor:
    """M uv points in radians per pixel: N(0, (pi/4)^2) per axis inside [-pi, pi)^2, outside the (0, 0) cell."""
    parts, need = [], M
    while need > 0:
        c = math.pi / 4 * torch.randn(need + need // 8 + 256, 2, generator=g, device=g.device, dtype=torch.float64)
        c = c[((c >= -math.pi) & (c < math.pi)).all(1) & (c.abs().amax(1) >= math.pi / n)][:need]
        parts.append(c)
        need -= c.shape[0]
    return torch.cat(parts).contiguous()


def _sources(g, n: int):
    """(amplitude, centre row, centre column, width) of blobs and point sources (width 0), centres from the image's middle pixel."""
    nb, npt = 3 + n // 128, 10 + n // 16
    blob = torch.stack([_uniform(g, 0.3, 1.0, nb), _uniform(g, -0.4 * n, 0.4 * n, nb), _uniform(g, -0.4 * n, 0.4 * n, nb),
                        _uniform(g, 1.5, max(1.6, n / 12), nb)], 1)
    flux = 0.1 * (1 - 0.99 * _uniform(g, 0.0, 1.0, npt)) ** -0.5
    at = torch.randint(-n // 2, n // 2, (npt, 2), generator=g, device=g.device).double()
    return torch.cat([blob, torch.cat([flux[:, None], at, torch.zeros_like(flux)[:, None]], 1)])


def _sky(src: torch.Tensor, n: int) -> torch.Tensor:
    p = torch.arange(n, device=src.device, dtype=torch.float64) - n // 2
    img = torch.zeros(n, n, device=src.device, dtype=torch.float64)
    for a, r, c, s in src[src[:, 3] > 0].tolist():
        img += a * torch.exp(-((p - r) ** 2) / (2 * s * s))[:, None] * torch.exp(-((p - c) ** 2) / (2 * s * s))[None, :]
    pts = src[src[:, 3] == 0]
    img.index_put_(((pts[:, 1] + n // 2).long(), (pts[:, 2] + n // 2).long()), pts[:, 0], accumulate=True)
    return img


def _measured(g, uv: torch.Tensor, n: int, src: torch.Tensor):
    """Noisy visibilities of the sources (their analytic transform) and the l2 bound on the noise."""
    y = torch.empty(uv.shape[0], dtype=torch.complex128, device=uv.device)
    amp = torch.where(src[:, 3] > 0, src[:, 0] * 2 * math.pi * src[:, 3] ** 2, src[:, 0])
    for lo in range(0, uv.shape[0], 1 << 18):
        u = uv[lo:lo + (1 << 18)]
        ph = (u @ src[:, 1:3].T).to(torch.float32)
        env = torch.exp((-(u * u).sum(1, keepdim=True) * (src[:, 3] ** 2)[None, :] / 2)).to(torch.float32) * amp.float()
        y[lo:lo + (1 << 18)] = torch.complex((env * torch.cos(ph)).sum(1), -(env * torch.sin(ph)).sum(1))
    M = uv.shape[0]
    sigma = float(torch.linalg.vector_norm(y)) / math.sqrt(M) * 10 ** (-30.0 / 20)
    noise = torch.randn(M, 2, generator=g, device=g.device, dtype=torch.float64)
    y = y + sigma / math.sqrt(2) * torch.view_as_complex(noise)
    return y, sigma * math.sqrt(M + 2 * math.sqrt(M))


def _types(case):
    return (torch.float32, torch.complex64) if case["prec"] == "fp32" else (torch.float64, torch.complex128)


def _inputs(case: dict, seed: int) -> dict:
    """The case's arrays on the device (the same for run and exact)."""
    g = _generator(seed)
    rt, ct = _types(case)
    op = case["op"]
    if op == "batch":
        parts = []
        for k, m in enumerate(_members(case)):
            parts.append(_inputs(dict(m, op="solve", blocks=1, prec=case["prec"]), seed * 1009 + k))
        return {"parts": parts}
    n = case["n"]
    if op == "sara_adj":
        q = bin(case["mask"]).count("1")
        return {"c": torch.randn(q, n, n, generator=g, device=g.device, dtype=torch.float64).to(rt)}
    src = _sources(g, n)
    if op == "sara_fwd":
        return {"x": _sky(src, n).to(rt)}
    uv = _coverage(g, case["M"], n)
    d = {"uv": uv}
    if op in ("phi", "gram"):
        d["x"] = _sky(src, n).to(rt)
    else:
        y, d["eps"] = _measured(g, uv, n, src)
        d["y"] = y.to(ct)
    if op == "solve":
        d["ids"] = torch.randint(0, case["blocks"], (case["M"],), generator=g, device=g.device, dtype=torch.int32)
    return d


def prepare(case: dict, seed: int):
    d = _inputs(case, seed)
    op = case["op"]
    if op in ("sara_fwd", "sara_adj"):
        # Psi comes with an operator; a token coverage serves
        o = binding.Operator(_coverage(_generator(seed), 64, case["n"]), case["n"], case["levels"], case["prec"])
        o.set_dictionary(case["mask"])
        return dict(d, case=case, o=o)
    if op == "batch":
        os = [binding.Operator(p["uv"], m["n"], case["levels"], case["prec"]) for p, m in zip(d["parts"], _members(case))]
        return dict(case=case, os=os, ys=[p["y"] for p in d["parts"]], eps=[p["eps"] for p in d["parts"]])
    if op == "image":
        host = {k: d[k].cpu() for k in ("uv", "y")}
        if torch.cuda.is_available():
            host = {k: v.pin_memory() for k, v in host.items()}
        return dict(host, case=case, eps=d["eps"])
    o = binding.Operator(d["uv"], case["n"], case.get("levels", 3), case["prec"])
    if op == "solve":
        if case["blocks"] > 1:
            o.set_blocks(d["ids"], case["blocks"])
        o.set_dictionary(case["mask"])
        o.set_prior(case["prior"], 20)
    if op == "gram" and case["mode"] == 1:
        o.gram(d["x"], 1)  # the composite is precomputed once per coverage
    return dict(d, case=case, o=o)


# ------------------------------------------------------------------ one pass
def _solved(r) -> dict:
    return {"x": r.x, "objective": r.stats["objective"], "residual": r.stats["residual"]}


def run(s):
    case = s["case"]
    op = case["op"]
    if op == "phi":
        return s["o"].phi(s["x"])
    if op == "phi_adj":
        return s["o"].phi_adj(s["y"])
    if op == "gram":
        return s["o"].gram(s["x"], case["mode"])
    if op == "sara_fwd":
        return s["o"].sara_fwd(s["x"])
    if op == "sara_adj":
        return s["o"].sara_adj(s["c"])
    if op == "solve":
        return _solved(s["o"].solve(s["y"], s["eps"], t_max=case["t_max"], n_reweight=case["n_reweight"]))
    if op == "batch":
        return [_solved(r) for r in binding.batch_solve(s["os"], s["ys"], s["eps"], t_max=case["t_max"])]
    return _solved(binding.solve_from_host(s["uv"], s["y"], case["n"], case["levels"], s["eps"], case["prec"],
                                           t_max=case["t_max"], n_reweight=case["n_reweight"]))


# ------------------------------------------------------------------ what a pass cannot do without
def _fft_flops(K: int) -> float:
    return 2.5 * K * K * 2 * math.log2(K)  # a real 2D transform of side K


def _sara_macs(mask: int, levels: int, N: int) -> float:
    taps = sum(2 * k for k in range(1, 9) if mask >> k & 1)
    return 2.0 * taps * N * sum(0.25 ** lev for lev in range(levels))


def work(case: dict) -> dict:
    r = 4 if case["prec"] == "fp32" else 8
    op = case["op"]
    if op == "batch":
        ws = [work(dict(m, op="solve", levels=case["levels"], prior="l1", mask=ALL_BASES, t_max=case["t_max"],
                        n_reweight=0, prec=case["prec"])) for m in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    n = case["n"]
    N, K = n * n, 2 * n
    if op in ("sara_fwd", "sara_adj"):
        q = bin(case["mask"]).count("1")
        return {"bytes": (1 + q) * N * r, "flops": 2 * _sara_macs(case["mask"], case["levels"], N)}
    M = case["M"]
    pair = 64 * 4.0 * M + _fft_flops(K)  # interpolation of M points and one transform
    conv = 2 * _fft_flops(K)
    if op in ("phi", "phi_adj"):  # image, positions (two coordinates), visibilities
        return {"bytes": N * r + 2 * M * r + 2 * M * r, "flops": pair}
    if op == "gram":
        if case["mode"] == 1:  # image in and out, the composite's half spectrum
            return {"bytes": 2 * N * r + (K // 2 + 1) * K * r, "flops": conv}
        return {"bytes": 2 * N * r + 2 * M * r, "flops": 2 * pair}
    # a solve, per SDMM iteration: 10 CG steps (the composite's spectrum; x, r, p in and out), the ball block
    # (positions, y, z_3 in and out), the prior's block (its dual in and out and its weights) and positivity
    q = bin(case.get("mask", ALL_BASES)).count("1") if case.get("prior", "l1") == "l1" else 3
    it = case["t_max"] * (1 + case["n_reweight"])
    per = 10 * (2 * N + 6 * N) * r + M * 8 * r + (3 * q + 4) * N * r
    fl = 11 * conv + 2 * pair
    fl += 4 * _sara_macs(case.get("mask", ALL_BASES), case["levels"], N) if case.get("prior", "l1") == "l1" else 20 * 20.0 * N
    return {"bytes": it * per + 16 * M + 2 * M * r + N * r, "flops": it * fl}


# ------------------------------------------------------------------ the same in 64 bits
_BETA = math.pi * math.sqrt((J / 2) ** 2 * 1.5 ** 2 - 0.8)


def _kb(s: torch.Tensor) -> torch.Tensor:
    a = (1 - (2 * s / J) ** 2)
    v = torch.special.i0(_BETA * torch.sqrt(a.clamp(min=0))) / torch.special.i0(torch.tensor(_BETA, dtype=torch.float64, device=s.device))
    return torch.where(a >= 0, v, torch.zeros_like(v))


class _Phi:
    """Phi and Re Phi^H as a Kaiser-Bessel NUFFT on the grid of side 2n."""

    def __init__(self, uv: torch.Tensor, n: int):
        self.uv, self.n, self.K, dev = uv, n, 2 * n, uv.device
        p = torch.arange(n, device=dev, dtype=torch.float64) - n // 2
        self.at = (p % self.K).long()
        d = _BETA ** 2 - (math.pi * J * p / self.K) ** 2  # positive over the image: the transform's sinh branch
        root = torch.sqrt(d)
        hat = torch.sinh(root) / root * J / torch.special.i0(torch.tensor(_BETA, dtype=torch.float64, device=dev))
        self.S = 1 / (hat[:, None] * hat[None, :])

    def _taps(self, lo):
        t = self.uv[lo:lo + (1 << 18)] * self.K / (2 * math.pi)
        j = t.floor().long()[:, :, None] + torch.arange(J, device=t.device) - J // 2 + 1
        w = _kb(t[:, :, None] - j)
        j = j % self.K
        return (j[:, 0, :, None] * self.K + j[:, 1, None, :]).reshape(t.shape[0], -1), (w[:, 0, :, None] * w[:, 1, None, :]).reshape(t.shape[0], -1)

    def phi(self, x):
        G = torch.zeros(self.K, self.K, dtype=torch.complex128, device=x.device)
        G[self.at[:, None], self.at[None, :]] = (self.S * x).to(torch.complex128)
        G = torch.fft.fft2(G).reshape(-1)
        parts = []
        for lo in range(0, self.uv.shape[0], 1 << 18):
            i, w = self._taps(lo)
            parts.append((G[i] * w).sum(1))
        return torch.cat(parts)

    def adj(self, y):
        G = torch.zeros(self.K * self.K, 2, dtype=torch.float64, device=y.device)
        for lo in range(0, self.uv.shape[0], 1 << 18):
            i, w = self._taps(lo)
            v = torch.view_as_real(w * y[lo:lo + (1 << 18), None]).reshape(-1, 2)
            G.index_add_(0, i.reshape(-1), v)
        g = torch.fft.ifft2(torch.view_as_complex(G).reshape(self.K, self.K)) * self.K ** 2
        return self.S * g[self.at[:, None], self.at[None, :]].real


class _Composite:
    """Re Phi^H Phi as a convolution with the even part of its point-spread function."""

    def __init__(self, uv, n):
        self.n, K = n, 2 * n
        psf = _Phi(uv, K).adj(torch.ones(uv.shape[0], dtype=torch.complex128, device=uv.device))
        self.khat = torch.fft.fft2(torch.roll(psf, (-n, -n), (0, 1))).real[:, :n + 1].contiguous()

    def __call__(self, x):
        K = 2 * self.n
        return torch.fft.irfft2(torch.fft.rfft2(x, s=(K, K)) * self.khat, s=(K, K))[:self.n, :self.n]


def _filters(k: int):
    """Minimum-phase Daubechies low-pass filter of k vanishing moments by spectral factorisation, and its mirror."""
    h = np.array([1.0 + 0j])
    for _ in range(k):
        h = np.convolve(h, [1.0, 1.0])
    if k > 1:
        for y in np.roots([math.comb(k - 1 + i, i) for i in range(k)][::-1]):
            b = 2 - 4 * y
            e = np.sqrt(b * b - 4 + 0j)
            z = (b + e) / 2 if abs(b + e) < 2 else (b - e) / 2
            h = np.convolve(h, [1.0, -z])
    h = h.real * (math.sqrt(2) / h.real.sum())
    return h.tolist(), [(-1) ** i * v for i, v in enumerate(h[::-1].tolist())]


def _split(x, h, g, dim):
    lo, hi = 0, 0
    for m in range(len(h)):
        s = torch.roll(x, -m, dim)
        s = s[::2] if dim == 0 else s[:, ::2]
        lo, hi = lo + h[m] * s, hi + g[m] * s
    return torch.cat([lo, hi], dim)


def _merge(c, h, g, dim):
    H = c.shape[dim] // 2
    x = torch.zeros_like(c)
    for m in range(len(h)):
        u = torch.zeros_like(c)
        v = h[m] * c.narrow(dim, 0, H) + g[m] * c.narrow(dim, H, H)
        if dim == 0:
            u[::2] = v
        else:
            u[:, ::2] = v
        x = x + torch.roll(u, m, dim)
    return x


class _Psi:
    def __init__(self, mask, levels):
        self.bases = [k for k in range(9) if mask >> k & 1]
        self.levels, self.f = levels, {k: _filters(k) for k in self.bases if k}

    def fwd(self, x):
        out = []
        for k in self.bases:
            c = x.clone()
            for lev in range(self.levels if k else 0):
                L = x.shape[0] >> lev
                c[:L, :L] = _split(_split(c[:L, :L], *self.f[k], 1), *self.f[k], 0)
            out.append(c)
        return torch.stack(out) / math.sqrt(len(self.bases))

    def adj(self, c):
        x = 0
        for k, b in zip(self.bases, c):
            b = b.clone()
            for lev in reversed(range(self.levels if k else 0)):
                L = b.shape[0] >> lev
                b[:L, :L] = _merge(_merge(b[:L, :L], *self.f[k], 0), *self.f[k], 1)
            x = x + b
        return x / math.sqrt(len(self.bases))


def _grad(x):
    g = torch.zeros(2, *x.shape, dtype=x.dtype, device=x.device)
    g[0, :-1] = x[1:] - x[:-1]
    g[1, :, :-1] = x[:, 1:] - x[:, :-1]
    return g


def _div(q):
    a, b = q[0].clone(), q[1].clone()
    a[-1], b[:, -1] = 0, 0
    d = a + b
    d[1:] -= a[:-1]
    d[:, 1:] -= b[:, :-1]
    return d


def _length(g):
    return torch.sqrt(g[0] ** 2 + g[1] ** 2)


def _solve_exact(d: dict, case: dict) -> dict:
    """SDMM with the reweighting loop on the case's inputs."""
    uv, y, n, eps = d["uv"], d["y"].to(torch.complex128), case["n"], d["eps"]
    tv = case["prior"] == "tv"
    phi, gram = _Phi(uv, n), _Composite(uv, n)
    psi = None if tv else _Psi(case["mask"], case["levels"])
    x = torch.full((n, n), 1.0 / n, dtype=torch.float64, device=uv.device)
    for _ in range(30):
        x = gram(x)
        lam = float(torch.linalg.vector_norm(x))
        x = x / lam
    nu = 1 / math.sqrt(lam)
    back = nu * nu * phi.adj(y)
    gamma = 1e-3 * float((back if tv else psi.fwd(back)).abs().max())
    blocks = [(d["ids"] == b).nonzero()[:, 0] for b in range(case["blocks"])]
    radii = [eps * math.sqrt(len(b) / len(y)) for b in blocks]

    def Q(v):
        return nu * nu * gram(v) + 2 * v

    xh = torch.zeros(n, n, dtype=torch.float64, device=uv.device)
    w, delta1 = 1.0, 0.0
    for rnd in range(case["n_reweight"] + 1):
        if rnd:
            a = _length(_grad(xh)) if tv else psi.fwd(xh)
            delta1 = (float(a.std(unbiased=False)) or 1.0) if rnd == 1 else delta1
            delta = max(0.1 ** (rnd - 1) * delta1, 1e-4 * delta1)
            w = delta / (delta + a.abs())
        xs = Q(xh)
        z1, z2, z3 = 0.0, 0.0, 0.0
        q = torch.zeros(2, n, n, dtype=torch.float64, device=uv.device)
        for _ in range(case["t_max"]):
            r = xs - Q(xh)
            p, rr = r, float((r * r).sum())
            for _ in range(10):
                Ap = Q(p)
                pAp = float((p * Ap).sum())
                a = rr / pAp if pAp > 0 else 0.0
                xh, r = xh + a * p, r - a * Ap
                new = float((r * r).sum())
                p, rr = r + (new / rr if rr > 0 else 0.0) * p, new
            c1 = xh if tv else psi.fwd(xh)
            v = c1 + z1
            if tv:
                for _ in range(20):
                    q = q + 0.125 * _grad(v + _div(q))
                    m = _length(q)
                    q = q * torch.where(m > gamma * w, gamma * w / m.clamp(min=1e-300), torch.ones_like(m))
                r1 = v + _div(q)
                objective = float((w * _length(_grad(xh))).sum())
            else:
                r1 = torch.sign(v) * (v.abs() - gamma * w).clamp(min=0)
                objective = float((w * c1.abs()).sum())
            z1 = v - r1
            x1 = r1 - z1 if tv else psi.adj(r1 - z1)
            v = xh + z2
            r2 = v.clamp(min=0)
            z2 = v - r2
            px = phi.phi(xh)
            v = nu * px + z3
            r3 = v.clone()
            for b, e in zip(blocks, radii):
                off = v[b] - nu * y[b]
                s = float(torch.linalg.vector_norm(off))
                if s > nu * e:
                    r3[b] = nu * y[b] + off * (nu * e / s)
            z3 = v - r3
            xs = x1 + (r2 - z2) + nu * phi.adj(r3 - z3)
    return {"x": xh, "objective": objective, "residual": float(torch.linalg.vector_norm(y - px))}


def exact(case: dict, seed: int):
    d = _inputs(case, seed)
    op = case["op"]
    if op == "phi":
        return _Phi(d["uv"], case["n"]).phi(d["x"].double())
    if op == "phi_adj":
        return _Phi(d["uv"], case["n"]).adj(d["y"].to(torch.complex128))
    if op == "gram":
        if case["mode"] == 1:
            return _Composite(d["uv"], case["n"])(d["x"].double())
        P = _Phi(d["uv"], case["n"])
        return P.adj(P.phi(d["x"].double()))
    if op == "sara_fwd":
        return _Psi(case["mask"], case["levels"]).fwd(d["x"].double())
    if op == "sara_adj":
        return _Psi(case["mask"], case["levels"]).adj(d["c"].double())
    if op == "batch":
        return [_solve_exact(p, dict(m, levels=case["levels"], prior="l1", mask=ALL_BASES, blocks=1, t_max=case["t_max"],
                                     n_reweight=0)) for p, m in zip(d["parts"], _members(case))]
    if op == "image":
        d["ids"] = torch.zeros(case["M"], dtype=torch.int32, device=d["uv"].device)
        case = dict(case, prior="l1", mask=ALL_BASES, blocks=1)
    return _solve_exact(d, case)
