"""Timed cases of the Faceted HyperSARA library: what a program that images with it has it do.

Every case goes through the public binding (`paper_2003_07358_gb300.fhs`): iterations of
Algorithm 2 (`fhs_pdfb_iter`) from the smallest problem to the large image, a batch of
uneven sub-cubes on concurrent lanes, the two variants of the data term (DDE kernels,
preconditioned duals), and the operators that programs call on their own (Phi, its
adjoint, the sparsity and low-rankness duals, the reweighting).

A case is a dict of plain values:
  op            : "iterate", "batch", "measure", "adjoint", "sparsity", "lowrank" or "reweight"
  n1, n2, L     : image rows, columns, channels of the sub-cube
  Q             : Q x Q spatial facets; overlap 10 %; window "triangular" or "sine"
  M, B          : visibilities per channel, data blocks per channel
  S_d           : side of the DDE kernels (0: none)
  n_sub         : forward-backward sub-iterations of the preconditioned duals (0: U = I)
  cubes, lanes, shape_seed : the batch, in place of the sizes
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2003_07358_gb300.fhs import Context, CubeParams

OVERLAP = 0.1
TAPS, BETA, LEVELS = 7, 2.34 * 7, 4
SIGMA_UV = math.pi / 4            # spread of the reference channel's uv points (rad/pixel)
N_BLOBS, N_POINTS = 24, 24        # sources of the sky
ISNR_DB = 30.0
TAU = 0.33
N_ANT, S_ANT = 8, 5               # antennas and their 5 x 5 patterns: 9 x 9 kernels per baseline
SIDES = (128, 192, 256, 384, 512, 768)       # sides of the batch's images (2^k and 3 * 2^m)
BATCH_PIXELS = 32_000_000         # channels times pixels of a drawn batch, at most
SMALL_M = 1000                    # visibilities per channel where the operator reads none


def _case(name, op, n1, L, Q, M, B, n2=None, window="triangular", S_d=0, n_sub=0):
    c = dict(op=op, n1=n1, n2=n2 or n1, L=L, Q=Q, window=window, M=M, B=B, S_d=S_d, n_sub=n_sub)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest problem of the test suite: every launch is short, the launches and
        # the gaps between them are the time
        _case("iterate tiny", "iterate", 64, 4, 1, 2000, 1),
        # a small survey field with apodised facets: many launches that do not fill the GPU
        _case("iterate faceted", "iterate", 256, 20, 4, 256 * 256 // 2, 2, window="sine"),
        # an ordinary wide-band sub-cube: 32 channels, dense coverage, 8 x 8 facets
        _case("iterate precision", "iterate", 1024, 32, 8, 1024 * 1024, 4),
        # the large image: grids, facets and coverage density of the 4096^2 workload, on four
        # of a sub-cube's sixteen channels (the host's visibility sort stays short)
        _case("iterate large", "iterate", 4096, 4, 16, 4096 * 4096 // 2, 8),
        # independent sub-cubes of uneven shapes side by side, sides 2^k and 3 * 2^m, odd
        # channel counts, more than 32 channels
        dict(name="batch uneven", op="batch", cubes=8, lanes=4, shape_seed=3048),
        # calibrated direction-dependent effects: 15 x 15 footprints
        _case("iterate dde", "iterate", 512, 16, 4, 512 * 512 // 2, 8, S_d=9),
        # preconditioned data duals (inverse sampling density)
        _case("iterate preconditioned", "iterate", 512, 12, 3, 512 * 512, 4, n_sub=20),
        # model visibilities of an image (residuals, data simulation); rows and columns differ
        _case("measure", "measure", 2048, 8, 1, 2048 * 1024, 4, n2=1024),
        # dirty image of a 3 * 2^m field with an odd channel count
        _case("adjoint", "adjoint", 768, 23, 1, int(0.59 * 768 * 768), 1),
        # the two priors' dual updates of a whole 16-channel sub-cube of the 4096^2 workload
        _case("sparsity duals", "sparsity", 4096, 16, 16, SMALL_M, 1),
        _case("low-rankness duals", "lowrank", 4096, 16, 16, SMALL_M, 1),
        # weights of a reweighting cycle, more than 32 channels, ragged 6 x 6 facets
        _case("reweight", "reweight", 512, 38, 6, SMALL_M, 1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("iterate", "iterate", "iterate", "batch", "measure", "adjoint", "sparsity", "lowrank", "reweight"))
    while op == "batch":
        case = dict(op=op, cubes=rng.randint(3, 8), lanes=rng.choice((1, 2, 4)), shape_seed=rng.randrange(1 << 20))
        if sum(c["L"] * c["n1"] * c["n2"] for c in _batch_shapes(case)) <= BATCH_PIXELS:
            return case
    data = op in ("iterate", "measure", "adjoint")
    while True:
        n1 = rng.choice((64, 96, 128, 192, 256, 384, 512, 768, 1024, 2048, 4096))
        n2 = rng.choice((n1, n1, n1, max(64, n1 // 2)))
        if n1 > 1536 and n2 % 3 == 0:
            continue
        L = _log_int(rng, 4, 48)
        M = int(rng.uniform(0.3, 2.0) * n1 * n2) if data else SMALL_M
        S_d = n_sub = 0
        if op == "iterate":
            kind = rng.random()
            if kind < 0.15:
                S_d = 9
            elif kind < 0.3:
                n_sub = rng.randint(5, 20)
        Q = rng.randint(1, min(16, n1 // 16, n2 // 16))
        pixels = L * n1 * n2
        if (n1 * n2 // (Q * Q) >= 4 * L and L * M <= (1 << 25) and L * M * (16 if S_d else 4 if n_sub else 1) <= (1 << 25)
                and pixels <= ((1 << 26) if op == "iterate" else (1 << 28))):
            break
    return _case("", op, n1, L, Q, M, rng.randint(1, 8) if data else 1, n2=n2,
                 window=rng.choice(("triangular", "sine")), S_d=S_d, n_sub=n_sub)


def _batch_shapes(case):
    """The cubes of a batch: sides, channels, facets, coverage and blocks drawn one by one
    (the largest side appears once at least)."""
    rng = random.Random(case["shape_seed"])
    out = []
    for k in range(case["cubes"]):
        n = rng.choice(SIDES) if k else SIDES[-1]
        L, Q, ratio, B = rng.randint(8, 48), rng.randint(1, 6), rng.uniform(0.3, 2.0), rng.randint(1, 4)
        out.append(_case("", "iterate", n, L, Q, int(ratio * n * n), B))
    return out


# ------------------------------------------------------------------ inputs
def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _generator(seed, what):
    g = torch.Generator(device=_device())
    g.manual_seed((seed * 1000003 + what) & 0x7FFFFFFFFFFF)
    return g


def _tile_bounds(n, Q):
    return [i * n // Q for i in range(Q + 1)]


def _facets_1d(n, Q):
    tb = _tile_bounds(n, Q)
    return [(tb[i] - (int(math.floor(OVERLAP * (tb[i + 1] - tb[i]))) if i else 0), tb[i + 1]) for i in range(Q)]


def _facets(case):
    """Pixel ranges (r0, r1, c0, c1) of the nuclear facets, row by row."""
    return [(r0, r1, c0, c1) for r0, r1 in _facets_1d(case["n1"], case["Q"]) for c0, c1 in _facets_1d(case["n2"], case["Q"])]


def _n_coef(n1, n2):
    total = n1 * n2
    for b in range(1, 9):
        r, c = n1, n2
        for _ in range(LEVELS):
            r, c = (r + 2 * b - 1) // 2, (c + 2 * b - 1) // 2
            total += 3 * r * c
        total += r * c
    return total


class _Inputs:
    """What a program has in hand for one sub-cube in the middle of a reconstruction, from
    the seed alone: uv coverage, parameters, noisy data, the iterate and the duals."""

    def __init__(self, case, seed):
        self.case = case
        dev = _device()
        n1, n2, L, Q, M, B = (case[k] for k in ("n1", "n2", "L", "Q", "M", "B"))
        self.dev, self.nu = dev, np.linspace(1.0, 2.0, L)
        # reference coverage, partitioned into radial blocks of equal count
        g = _generator(seed, 1)
        base = torch.empty((0, 2), device=dev)
        while base.shape[0] < M:
            d = torch.randn((2 * M + 64, 2), generator=g, device=dev) * SIGMA_UV
            base = torch.cat([base, d[d.abs().amax(1) * self.nu[-1] < math.pi * (1 - 1e-5)]])
        base = base[:M]
        rank = torch.empty(M, dtype=torch.int64, device=dev)
        rank[torch.argsort((base * base).sum(1), stable=True)] = torch.arange(M, device=dev)
        bounds = [round(b * M / B) for b in range(B + 1)]
        block = torch.bucketize(rank, torch.tensor(bounds[1:-1], device=dev, dtype=torch.int64), right=True)
        self.order = torch.argsort(block, stable=True)
        base = base[self.order]
        self.uv = torch.cat([base * float(f) for f in self.nu])               # [L M][2], channel by channel
        self.M_lb = np.tile(np.diff(bounds).astype(np.int64), (L, 1))
        # sky: Gaussian blobs and points with power-law spectra
        g = _generator(seed, 2)
        ns = N_BLOBS + N_POINTS
        u = torch.rand((5, ns), generator=g, device=dev)
        self.amp, index = 0.1 + 0.9 * u[2], 2.0 * u[3] - 1.0
        self.pos_r, self.pos_c = n1 * (0.1 + 0.8 * u[0]), n2 * (0.1 + 0.8 * u[1])
        self.pos_r[N_BLOBS:], self.pos_c[N_BLOBS:] = self.pos_r[N_BLOBS:].floor(), self.pos_c[N_BLOBS:].floor()
        self.width = 1.0 + 3.0 * u[4]
        self.flux = [self.amp * torch.exp(index * math.log(f)) for f in self.nu]
        # parameters: operator norms from the sampling density, the noise-based heuristics
        gain = 4.0 if case["S_d"] else 1.0
        dens = [M / (2 * math.pi * (SIGMA_UV * f) ** 2) / 0.9 for f in self.nu]
        opn = np.array([3.0 * gain * (2 * math.pi) ** 2 * max(d, 4.0 * n1 * n2 / (2 * math.pi) ** 2 / 8) for d in dens])
        self.eta = np.full(L, 1.0 / (6.0 * n1 * n2)) if case["n_sub"] else 1.0 / opn
        power = float((self.amp ** 2).sum())
        self.sigma = np.full(L, math.sqrt(power) * 10 ** (-ISNR_DB / 20))
        sbar = math.sqrt(float(np.mean(self.sigma ** 2 / opn)))
        mchi = math.sqrt(2) * math.exp(math.lgamma((L + 1) / 2) - math.lgamma(L / 2))
        self.mu = sbar * (mchi + math.sqrt(max(L - mchi * mchi, 0.0)))
        self.facets = _facets(case)
        npix = [(r1 - r0) * (c1 - c0) for r0, r1, c0, c1 in self.facets]
        self.mu_bar = np.array([sbar * math.sqrt(p * L / min(p, L)) for p in npix])
        self.eps = np.sqrt(self.sigma[:, None] ** 2 * (M + 2 * math.sqrt(M)) * self.M_lb / M)

    def params(self):
        c = self.case
        return CubeParams(n1=c["n1"], n2=c["n2"], L=c["L"], Qy=c["Q"], Qx=c["Q"], overlap=OVERLAP, window=c["window"],
                          M_lb=self.M_lb, uv=self.uv.cpu().numpy(), eta=self.eta, mu=self.mu, mu_bar=self.mu_bar,
                          eps=self.eps, tau=TAU)

    def image(self, seed, what, noise):
        """[L][n1][n2]: the sky with relative errors and a non-negative background."""
        c = self.case
        g = _generator(seed, what)
        r = torch.arange(c["n1"], device=self.dev, dtype=torch.float32)[:, None]
        k = torch.arange(c["n2"], device=self.dev, dtype=torch.float32)[None, :]
        rows = torch.exp(-(r - self.pos_r) ** 2 / (2 * self.width ** 2))           # [n1][sources]
        cols = torch.exp(-(k - self.pos_c[:, None]) ** 2 / (2 * self.width[:, None] ** 2))
        rows[:, N_BLOBS:] = (r == self.pos_r[N_BLOBS:]).float()
        cols[N_BLOBS:] = (k == self.pos_c[N_BLOBS:, None]).float()
        out = torch.empty((c["L"], c["n1"], c["n2"]), device=self.dev)
        for l, flux in enumerate(self.flux):
            torch.matmul(rows * flux, cols, out=out[l])
            z = torch.randn((c["n1"], c["n2"]), generator=g, device=self.dev)
            out[l] = (out[l] * (1.0 + noise * z) + 0.01 * noise * z.abs()).clamp_(min=0.0)
        return out

    def visibilities(self):
        """Noiseless visibilities of the sky (closed form), complex64, caller's order."""
        c = self.case
        out = torch.empty(self.uv.shape[0], dtype=torch.complex64, device=self.dev)
        M = c["M"]
        for l, flux in enumerate(self.flux):
            uv = self.uv[l * M:(l + 1) * M]
            w2 = (uv * uv).sum(1)
            re, im = torch.zeros(M, device=self.dev), torch.zeros(M, device=self.dev)
            for s in range(N_BLOBS + N_POINTS):
                ph = uv[:, 0] * (self.pos_c[s] - c["n2"] // 2) + uv[:, 1] * (self.pos_r[s] - c["n1"] // 2)
                a = flux[s]
                if s < N_BLOBS:
                    a = a * 2 * math.pi * self.width[s] ** 2 * torch.exp(-0.5 * self.width[s] ** 2 * w2)
                re += a * torch.cos(ph)
                im -= a * torch.sin(ph)
            out[l * M:(l + 1) * M] = torch.complex(re, im)
        return out

    def complex_noise(self, seed, what, scale):
        g = _generator(seed, what)
        return torch.view_as_complex(torch.randn((self.uv.shape[0], 2), generator=g, device=self.dev) * (scale * math.sqrt(0.5)))

    def state(self, seed):
        """Iterate, duals and weights (caller's visibility order)."""
        c = self.case
        L, N, Q2 = c["L"], c["n1"] * c["n2"], c["Q"] ** 2
        s = self.priors(seed)
        clean = self.visibilities()
        sig = float(self.sigma[0])
        s.update(X=self.image(seed, 3, 0.05), Xcheck=self.image(seed, 4, 0.06),
                 y=clean + self.complex_noise(seed, 5, sig), u_prev=clean * 0.98 + self.complex_noise(seed, 6, 0.3 * sig),
                 v=self.complex_noise(seed, 7, 0.5 * sig))
        return s

    def priors(self, seed):
        """Prior duals W, P and weights theta, theta_bar."""
        c = self.case
        L = c["L"]
        I = _n_coef(c["n1"], c["n2"])
        g = _generator(seed, 8)
        W = torch.randn(L * I, generator=g, device=self.dev).mul_(0.3 * self.mu / math.sqrt(L))
        theta = torch.rand(I, generator=g, device=self.dev).mul_(0.95).add_(0.05)
        P = []
        for (r0, r1, c0, c1), m in zip(self.facets, self.mu_bar):
            n = (r1 - r0) * (c1 - c0)
            P.append(torch.randn(L * n, generator=g, device=self.dev).mul_(0.3 * m / math.sqrt(n)))
        theta_bar = torch.rand((len(P), L), generator=g, device=self.dev).mul_(0.95).add_(0.05).sort(dim=1).values
        return dict(W=W, theta=theta, P=torch.cat(P), theta_bar=theta_bar.reshape(-1).contiguous())

    def dde(self, seed):
        """Per-baseline kernels (products of antenna patterns) and each visibility's kernel."""
        c = self.case
        L, M = c["L"], c["M"]
        rng = np.random.default_rng(seed + 17)
        pairs = [(a, b) for a in range(N_ANT) for b in range(a + 1, N_ANT)]
        bl = rng.integers(0, len(pairs), size=M)[self.order.cpu().numpy()]
        R = S_ANT // 2
        j = np.arange(-R, R + 1)
        taper = 0.05 * np.exp(-(j[:, None] ** 2 + j[None, :] ** 2) / 2.0)
        S = 2 * S_ANT - 1
        kern = np.zeros((L, len(pairs), S, S), dtype=np.complex128)
        for l in range(L):
            d = rng.standard_normal((N_ANT, S_ANT, S_ANT, 2))
            d = (d[..., 0] + 1j * d[..., 1]) * taper
            d[:, R, R] = 1.0
            for k, (a, b) in enumerate(pairs):
                db = np.conj(d[b][::-1, ::-1])
                for r in range(S_ANT):
                    for q in range(S_ANT):
                        kern[l, k, r:r + S_ANT, q:q + S_ANT] += d[a][r, q] * db
        kidx = (np.arange(L)[:, None] * len(pairs) + bl[None, :]).astype(np.int32).ravel()
        return kern.reshape(-1, S, S).astype(np.complex64), kidx


def _cube_seed(seed, k):
    return seed * 64 + k


def _device_iterate(ctx, cube, s):
    """The arrays of one cube as fhs_pdfb_iter takes them (visibilities in internal order)."""
    vis = {}
    for k in ("y", "v", "u_prev"):
        vis[k] = torch.empty_like(s[k])
        ctx.fhs_vis_to_internal(cube, s[k], vis[k])
    state = {k: s[k] for k in ("W", "theta", "P", "theta_bar")}
    return {"X": s["X"], "Xcheck": s["Xcheck"], "y": vis["y"], "state": dict(state, v=vis["v"], u_prev=vis["u_prev"])}


def prepare(case, seed):
    op = case["op"]
    shapes = _batch_shapes(case) if op == "batch" else [case]
    inputs = [_Inputs(c, _cube_seed(seed, k)) for k, c in enumerate(shapes)]
    ctx = Context([i.params() for i in inputs])
    st = {"op": op, "ctx": ctx}
    if op in ("iterate", "batch"):
        st["iterates"] = []
        for k, i in enumerate(inputs):
            if i.case["S_d"]:
                ctx.fhs_set_dde(k, *i.dde(_cube_seed(seed, k)))
            if i.case["n_sub"]:
                ctx.fhs_set_preconditioning(k, i.case["n_sub"])
            st["iterates"].append(_device_iterate(ctx, k, i.state(_cube_seed(seed, k))))
        if op == "batch":
            ctx.fhs_set_lanes(case["lanes"])
        return st
    i, s0 = inputs[0], _cube_seed(seed, 0)
    if op == "measure":
        st["x"] = i.image(s0, 3, 0.05)
        st["internal"] = torch.empty(i.uv.shape[0], dtype=torch.complex64, device="cuda")
        st["y"] = torch.empty_like(st["internal"])
    elif op == "adjoint":
        v = i.visibilities() + i.complex_noise(s0, 5, float(i.sigma[0]))
        st["v"] = torch.empty_like(v)
        ctx.fhs_vis_to_internal(0, v, st["v"])
        st["x"] = torch.empty((case["L"], case["n1"], case["n2"]), device="cuda")
    else:
        st["x"] = i.image(s0, 3, 0.05)
        if op == "reweight":
            st["theta"] = torch.empty(_n_coef(case["n1"], case["n2"]), device="cuda")
            st["theta_bar"] = torch.empty(case["Q"] ** 2 * case["L"], device="cuda")
        else:
            s = i.priors(s0)
            keep = ("W", "theta") if op == "sparsity" else ("P", "theta_bar")
            st.update({k: s[k] for k in keep})
            st["A"] = i.image(s0, 9, 0.05)
    return st


def run(st):
    ctx, op = st["ctx"], st["op"]
    if op in ("iterate", "batch"):
        ctx.fhs_pdfb_iter(st["iterates"], 1, want_stats=False)
        return [dict(X=a["X"], Xcheck=a["Xcheck"], W=a["state"]["W"], P=a["state"]["P"], v=a["state"]["v"],
                     u_prev=a["state"]["u_prev"]) for a in st["iterates"]]
    if op == "measure":
        ctx.fhs_measure(0, st["x"], st["internal"])
        ctx.fhs_vis_to_user(0, st["internal"], st["y"])
        return {"y": st["y"]}
    if op == "adjoint":
        ctx.fhs_adjoint(0, st["v"], st["x"])
        return {"x": st["x"]}
    if op == "sparsity":
        ctx.fhs_prox_l21_sara_facets(0, st["x"], st["W"], st["theta"], st["A"])
        return {"W": st["W"], "A": st["A"]}
    if op == "lowrank":
        ctx.fhs_prox_nuclear_facets(0, st["x"], st["P"], st["theta_bar"], st["A"])
        return {"P": st["P"], "A": st["A"]}
    ctx.fhs_reweight(0, st["x"], st["theta"], st["theta_bar"])
    return {"theta": st["theta"], "theta_bar": st["theta_bar"]}


def work(case):
    """Bytes: every array of the call read once and, where it changes, written once (the
    visibilities' coordinates among them); no transform grids or wavelet bands in between.
    Operations: the two transforms and their 7 x 7 (or DDE) footprints, the wavelet
    filters, the facet Grams and products."""
    if case["op"] == "batch":
        parts = [work(c) for c in _batch_shapes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    op, n1, n2, L, M = case["op"], case["n1"], case["n2"], case["L"], case["M"]
    N, I, V = n1 * n2, _n_coef(n1, n2), L * M
    NF = sum((r1 - r0) * (c1 - c0) for r0, r1, c0, c1 in _facets(case))
    F = TAPS + (case["S_d"] - 1 if case["S_d"] else 0)
    fft = L * 5.0 * 4 * N * math.log2(4.0 * N) / 2          # real image: half of the complex transform
    foot = V * F * F * (8.0 if case["S_d"] else 4.0)
    filt = sum(2 * 2 * b * 2 * 2 * N * 4.0 / 3 for b in range(1, 9)) * L      # one direction
    nuc = L * NF * (4.0 * L + 4)
    if op == "measure":
        return {"bytes": 4 * N * L + 8 * V + 8 * V, "flops": fft + foot}
    if op == "adjoint":
        return {"bytes": 4 * N * L + 8 * V + 8 * V, "flops": fft + foot}
    if op == "sparsity":
        return {"bytes": 4 * N * L + 8 * I * L + 4 * I + 8 * N * L, "flops": 2 * filt + 6.0 * I * L}
    if op == "lowrank":
        return {"bytes": 4 * N * L + 8 * NF * L + 8 * N * L, "flops": nuc}
    if op == "reweight":
        return {"bytes": 4 * N * L + 4 * I + 4 * L * case["Q"] ** 2, "flops": filt + 2.0 * I * L + L * NF * 2.0 * L}
    return {"bytes": 16 * N * L + 8 * I * L + 4 * I + 8 * NF * L + V * (8 + 1 + 8 + 16 + 16),
            "flops": 2 * fft + 2 * foot + 2 * filt + 6.0 * I * L + nuc + V * (20.0 + 12.0 * case["n_sub"])}


# ---------------------------------------------- the same results in 64 bits
def _i0(x):
    """Modified Bessel function I0 by its power series (x up to BETA)."""
    q, t, s = x * x / 4.0, torch.ones_like(x), torch.ones_like(x)
    for k in range(1, 60):
        t = t * q / (k * k)
        s = s + t
    return s


def _taps64(om, K):
    """First tap and the 7 Kaiser-Bessel weights of every coordinate."""
    t = om.double() * (K / (2.0 * math.pi))
    k0 = torch.floor(t - TAPS / 2.0).long() + 1
    u = (t - k0)[:, None] - torch.arange(TAPS, device=om.device)
    arg = 1.0 - (2.0 * u / TAPS) ** 2
    w = torch.where(arg >= 0, _i0(BETA * arg.clamp(min=0).sqrt()), torch.zeros_like(arg))
    return k0, w / _i0(torch.tensor(BETA, dtype=torch.float64, device=om.device))


def _scale64(n, dev):
    theta = math.pi * (torch.arange(n, dtype=torch.float64, device=dev) - n // 2) / n
    z = torch.sqrt(BETA ** 2 - (TAPS * theta / 2.0) ** 2)
    return _i0(torch.tensor(BETA, dtype=torch.float64, device=dev)) * z / (TAPS * torch.sinh(z))


class _Phi64:
    """Phi_l of one sub-cube and its adjoint, channel by channel."""

    def __init__(self, inp, kern=None, kidx=None):
        self.inp, c = inp, inp.case
        self.n1, self.n2, self.M = c["n1"], c["n2"], c["M"]
        dev = inp.dev
        self.K1, self.K2 = 2 * self.n1, 2 * self.n2
        self.s = _scale64(self.n1, dev)[:, None] * _scale64(self.n2, dev)[None, :]
        self.rows = (torch.arange(self.n1, device=dev) - self.n1 // 2) % self.K1
        self.cols = (torch.arange(self.n2, device=dev) - self.n2 // 2) % self.K2
        self.kern = None if kern is None else torch.as_tensor(kern, device=dev).to(torch.complex128)
        self.kidx = None if kidx is None else torch.as_tensor(kidx, device=dev).long()

    def _footprints(self, l):
        """(slice, flat cells [m][F F], weights [m][F F]) of the channel in pieces."""
        step = 1 << (16 if self.kern is not None else 19)
        for a in range(0, self.M, step):
            m = slice(l * self.M + a, l * self.M + min(a + step, self.M))
            uv = self.inp.uv[m]
            kr, wr = _taps64(uv[:, 1], self.K1)
            kc, wc = _taps64(uv[:, 0], self.K2)
            F = TAPS
            if self.kern is None:
                w = wr[:, :, None] * wc[:, None, :]
            else:
                S = self.kern.shape[1]
                F = TAPS + S - 1
                br = torch.zeros((uv.shape[0], S, F), dtype=torch.complex128, device=uv.device)
                bc = torch.zeros_like(br)
                for j in range(S):
                    br[:, j, j:j + TAPS] = wr.to(torch.complex128)
                    bc[:, j, j:j + TAPS] = wc.to(torch.complex128)
                w = br.transpose(1, 2) @ (self.kern[self.kidx[m]] @ bc)
                kr, kc = kr - S // 2, kc - S // 2
            k = torch.arange(F, device=uv.device)
            cell = ((kr[:, None] + k) % self.K1)[:, :, None] * self.K2 + ((kc[:, None] + k) % self.K2)[:, None, :]
            yield m, cell.reshape(uv.shape[0], -1), w.reshape(uv.shape[0], -1)

    def measure(self, x):
        out = torch.empty(self.inp.uv.shape[0], dtype=torch.complex128, device=x.device)
        for l in range(x.shape[0]):
            g = torch.zeros((self.K1, self.K2), dtype=torch.complex128, device=x.device)
            g[self.rows[:, None], self.cols[None, :]] = (self.s * x[l].double()).to(torch.complex128)
            g = torch.fft.fft2(g).reshape(-1)
            for m, cell, w in self._footprints(l):
                out[m] = (g[cell] * w).sum(1)
        return out

    def adjoint(self, v):
        L = self.inp.case["L"]
        out = torch.empty((L, self.n1, self.n2), dtype=torch.float64, device=v.device)
        for l in range(L):
            g = torch.zeros((self.K1 * self.K2, 2), dtype=torch.float64, device=v.device)
            for m, cell, w in self._footprints(l):
                g.index_add_(0, cell.reshape(-1), torch.view_as_real((w.conj() * v[m].to(torch.complex128)[:, None]).reshape(-1)))
            f = torch.fft.ifft2(torch.view_as_complex(g).reshape(self.K1, self.K2), norm="forward")
            out[l] = self.s * f[self.rows[:, None], self.cols[None, :]].real
        return out


def _daubechies64():
    out = []
    for N in range(1, 9):
        poly = np.array([1.0 + 0j])
        for y in (np.roots([math.comb(N - 1 + k, k) for k in range(N)][::-1]) if N > 1 else []):
            b = 2.0 - 4.0 * y
            z = (b + np.sqrt(b * b - 4.0 + 0j)) / 2.0
            poly = np.convolve(poly, [1.0, -(z if abs(z) < 1.0 else b - z)])
        for _ in range(N):
            poly = np.convolve(poly, [1.0, 1.0])
        h = poly.real * (math.sqrt(2.0) / poly.real.sum())
        out.append((h, [(-1) ** k * h[2 * N - 1 - k] for k in range(2 * N)]))
    return out


def _down(a, f, axis):
    """c[k] = sum_t f[t] a[2k + 1 - t] along the axis, zero outside the signal."""
    m, F = a.shape[axis], len(f)
    n = (m + F - 1) // 2
    p = torch.nn.functional.pad(a, (F, F) if axis == -1 else (0, 0, F, F))
    out = 0
    for t in range(F):
        i = F + 1 - t
        out = out + f[t] * (p[..., i:i + 2 * n:2] if axis == -1 else p[..., i:i + 2 * n:2, :])
    return out


def _up(c, f, m, axis):
    """Transpose of _down: a[i] = sum_k f[2k + 1 - i] c[k], i < m."""
    n, F = c.shape[axis], len(f)
    shape = list(c.shape)
    shape[axis] = 2 * n + 2 * F
    a = torch.zeros(shape, dtype=c.dtype, device=c.device)
    for t in range(F):
        i = F + 1 - t
        (a[..., i:i + 2 * n:2] if axis == -1 else a[..., i:i + 2 * n:2, :]).add_(c, alpha=f[t])
    return a[..., F:F + m] if axis == -1 else a[..., F:F + m, :]


def _analysis64(x):
    """Psi^dagger x of one channel [n1][n2] -> [I]."""
    parts = []
    for h, g in _daubechies64():
        a = x
        for _ in range(LEVELS):
            lx, hx = _down(a, h, -1), _down(a, g, -1)
            parts += [_down(hx, h, -2).reshape(-1), _down(lx, g, -2).reshape(-1), _down(hx, g, -2).reshape(-1)]
            a = _down(lx, h, -2)
        parts.append(a.reshape(-1))
    return torch.cat(parts + [x.reshape(-1)]) / 3.0


def _synthesis64(w, n1, n2):
    out, off = torch.zeros((n1, n2), dtype=torch.float64, device=w.device), 0
    for h, g in _daubechies64():
        sizes, bands = [(n1, n2)], []
        for _ in range(LEVELS):
            r, c = ((s + len(h) - 1) // 2 for s in sizes[-1])
            sizes.append((r, c))
            bands.append([w[off + k * r * c:off + (k + 1) * r * c].reshape(r, c) for k in range(3)])
            off += 3 * r * c
        a = w[off:off + r * c].reshape(r, c)
        off += r * c
        for j in range(LEVELS, 0, -1):
            m1, m2 = sizes[j - 1]
            d0, d1, d2 = bands[j - 1]
            lx = _up(a, h, m1, -2) + _up(d1, g, m1, -2)
            hx = _up(d0, h, m1, -2) + _up(d2, g, m1, -2)
            a = _up(lx, h, m2, -1) + _up(hx, g, m2, -1)
        out += a
    return (out + w[off:].reshape(n1, n2)) / 3.0


def _sparsity64(inp, x, W, theta):
    """W <- Z min(1, mu theta / ||Z||), Z = W + Psi^dagger x, and Psi W."""
    L, n1, n2 = x.shape
    Z = W.reshape(L, -1).double()
    for l in range(L):
        Z[l] += _analysis64(x[l].double())
    norm = torch.zeros_like(Z[0])
    for l in range(L):
        norm += Z[l] ** 2
    Z *= (inp.mu * theta.double() / norm.sqrt().clamp(min=1e-300)).clamp(max=1.0)
    return Z.reshape(-1), torch.stack([_synthesis64(Z[l], n1, n2) for l in range(L)])


def _window64(case, n, dev):
    out, f = [], _facets_1d(n, case["Q"])
    tb = _tile_bounds(n, case["Q"])
    for i, (a, b) in enumerate(f):
        w = torch.ones(b - a, dtype=torch.float64, device=dev)
        for o, at, flip in ((tb[i] - a, 0, False), (tb[i + 1] - f[i + 1][0] if i + 1 < len(f) else 0, None, True)):
            if o:
                r = (torch.arange(o, dtype=torch.float64, device=dev) + 1) / (o + 1)
                r = torch.sin(math.pi / 2 * r) ** 2 if case["window"] == "sine" else r
                if flip:
                    w[b - a - o:] = 1 - r
                else:
                    w[:o] = r
        out.append(w)
    return out


def _facet_matrices64(inp, x):
    c = inp.case
    wy, wx = _window64(c, c["n1"], inp.dev), _window64(c, c["n2"], inp.dev)
    for q, (r0, r1, c0, c1) in enumerate(inp.facets):
        D = wy[q // c["Q"]][:, None] * wx[q % c["Q"]][None, :]
        yield q, (r0, r1, c0, c1), D, x[:, r0:r1, c0:c1].double() * D


def _lowrank64(inp, x, P, theta_bar):
    """P <- Z V diag(min(1, mu_bar theta_bar / s)) V^T, Z = P + D x, and sum_q D P."""
    L = x.shape[0]
    theta_bar = theta_bar.reshape(-1, L).double()
    A, out, off = torch.zeros(x.shape, dtype=torch.float64, device=x.device), [], 0
    for q, (r0, r1, c0, c1), D, DX in _facet_matrices64(inp, x):
        n = D.numel()
        Z = P[off:off + L * n].reshape(L, n).double() + DX.reshape(L, n)
        off += L * n
        lam, V = torch.linalg.eigh((Z @ Z.T).cpu())
        s, V = lam.clamp(min=0).sqrt().flip(0).to(x.device), V.flip(1).to(x.device)
        m = (float(inp.mu_bar[q]) * theta_bar[q] / s.clamp(min=1e-300)).clamp(max=1.0)
        Pn = ((V * m) @ V.T) @ Z
        out.append(Pn.reshape(-1))
        A[:, r0:r1, c0:c1] += D * Pn.reshape(DX.shape)
    return torch.cat(out), A


def _data64(inp, s, phi):
    """New data duals v and eta Re Phi^dagger v (Euclidean or preconditioned projections)."""
    c = inp.case
    u = phi.measure(s["X"])
    y, v, z = s["y"].to(torch.complex128), s["v"].to(torch.complex128), 2 * u - s["u_prev"].to(torch.complex128)
    off = 0
    for l in range(c["L"]):
        if c["n_sub"]:
            uv = inp.uv[l * c["M"]:(l + 1) * c["M"]].double()
            cell = (torch.floor(uv[:, 1] * c["n1"] / math.pi + 0.5).long() % (2 * c["n1"])) * (2 * c["n2"]) \
                + torch.floor(uv[:, 0] * c["n2"] / math.pi + 0.5).long() % (2 * c["n2"])
            U_l = 1.0 / torch.bincount(cell)[cell].double()
        for m, eps in zip(inp.M_lb[l], inp.eps[l]):
            b = slice(off, off + int(m))

            def inside(d):
                return d * min(1.0, float(eps) / float(torch.linalg.vector_norm(d)))

            if c["n_sub"]:
                U = U_l[off - l * c["M"]:off - l * c["M"] + int(m)]
                d = v[b] / U + z[b] - y[b]
                w, g = inside(d), 1.0 / float(U.max())
                for _ in range(c["n_sub"]):
                    w = inside(w - g * U * (w - d))
                v[b] = U * (d - w)
            else:
                d = v[b] + z[b] - y[b]
                v[b] = d - inside(d)
            off += int(m)
    return phi.adjoint(v) * torch.as_tensor(inp.eta, device=u.device)[:, None, None]


def _iterate64(inp, seed):
    s = inp.state(seed)
    phi = _Phi64(inp, *(inp.dde(seed) if inp.case["S_d"] else ()))
    A = _data64(inp, s, phi)
    W, Aw = _sparsity64(inp, s["Xcheck"], s["W"], s["theta"])
    A += Aw
    P, Ap = _lowrank64(inp, s["Xcheck"], s["P"], s["theta_bar"])
    A += Ap
    X0 = s["X"].double()
    X = (X0 - TAU * A).clamp(min=0.0)
    return dict(X=X, Xcheck=2 * X - X0, W=W, P=P, v=None, u_prev=None)      # v, u_prev: the library's own order


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        return [_iterate64(_Inputs(c, _cube_seed(seed, k)), _cube_seed(seed, k)) for k, c in enumerate(_batch_shapes(case))]
    s0 = _cube_seed(seed, 0)
    inp = _Inputs(case, s0)
    if op == "iterate":
        return [_iterate64(inp, s0)]
    if op == "measure":
        return {"y": _Phi64(inp).measure(inp.image(s0, 3, 0.05))}
    if op == "adjoint":
        return {"x": _Phi64(inp).adjoint(inp.visibilities() + inp.complex_noise(s0, 5, float(inp.sigma[0])))}
    x = inp.image(s0, 3, 0.05)
    if op == "reweight":
        L = case["L"]
        norm = sum(_analysis64(x[l].double()) ** 2 for l in range(L)).sqrt()
        bars = []
        for q, _, D, DX in _facet_matrices64(inp, x):
            Z = DX.reshape(L, -1)
            s = torch.linalg.eigvalsh((Z @ Z.T).cpu()).clamp(min=0).sqrt().flip(0)
            bars.append(float(inp.mu_bar[q]) / (s + float(inp.mu_bar[q])))
        return {"theta": inp.mu / (norm + inp.mu), "theta_bar": torch.cat(bars)}
    s, A = inp.priors(s0), inp.image(s0, 9, 0.05).double()
    if op == "sparsity":
        W, Aw = _sparsity64(inp, x, s["W"], s["theta"])
        return {"W": W, "A": A + Aw}
    P, Ap = _lowrank64(inp, x, s["P"], s["theta_bar"])
    return {"P": P, "A": A + Ap}
