"""What is timed: the work a user of the library has it do, through its public entry points.

Every case is one call (or one pair of calls, one gradient, one run of
iterations) on a problem of the paper's kind: an L-channel image cube, a
Gaussian-density uv coverage scaled with the channel frequency, and priors on
the whole cube. `listed` gives the sizes of the repository's own workloads and
tests and the corners beside them (the smallest grids, sides that are not
powers of two, ragged and empty channels, FP64, weights, data blocks); `draw`
gives others of the same ranges. `exact` restates every case in 64-bit torch
expressions from the definitions, on the same inputs.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_1806_04596_gb300 import autograd as hsg
from paper_1806_04596_gb300 import hypersara as hs

J = 8                                                          # support of the interpolation kernel
BETA = math.pi * math.sqrt((J / 2.0) ** 2 * 1.5 ** 2 - 0.8)     # its shape at oversampling 2


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest problem of the tests and the latency end of the operators: 64 x 64, FP64, one
        # forward and one adjoint, where launches are what is paid for
        dict(name="phi_pair_64_f64", kind="phi_pair", nx=64, ny=64, L=4, M=2000, prec="f64", ragged=False,
             weights=False, compensated=False),
        # the benchmarked 256 x 256, 60-channel problem: predicted visibilities of a model cube
        dict(name="phi_fwd_256", kind="phi_fwd", nx=256, ny=256, L=60, M=32768, prec="f32", ragged=False,
             weights=False, compensated=False),
        # the same problem: the dirty cube / the gradient of the data term
        dict(name="phi_adj_256", kind="phi_adj", nx=256, ny=256, L=60, M=32768, prec="f32", ragged=False,
             weights=False, compensated=False),
        # the large image of the precision workload with natural weights, forward and adjoint
        dict(name="phi_pair_1024_w", kind="phi_pair", nx=1024, ny=1024, L=16, M=200_000, prec="f32", ragged=False,
             weights=True, compensated=False),
        # sides 5 2^a and 3 2^a, uneven channels and an empty one, as flagged data leave them
        dict(name="phi_pair_640x384_ragged", kind="phi_pair", nx=640, ny=384, L=7, M=45_001, prec="f32", ragged=True,
             weights=False, compensated=False),
        # analysis of a large cube (re-weighting, objective values)
        dict(name="psi_fwd_1024", kind="psi_fwd", nx=1024, ny=1024, L=16, prec="f32"),
        # synthesis on the benchmarked cube
        dict(name="psi_adj_256", kind="psi_adj", nx=256, ny=256, L=60, prec="f32"),
        # joint-sparsity prior with re-weighted rows on the benchmarked cube, dual form
        dict(name="l21_256_w", kind="l21", nx=256, ny=256, L=60, prec="f32", dual=True, weights=True),
        # low-rank prior alone (no warm start), prox form
        dict(name="nuclear_256", kind="nuclear", nx=256, ny=256, L=60, prec="f32", dual=False),
        # differentiable objective and its gradient at the 512 x 512, 32-channel workload's image size
        dict(name="grad_512", kind="grad", nx=512, ny=512, L=32, M=100_000, prec="f32", ragged=True),
        # the solver itself: ten iterations of the benchmarked problem, the image and the diagnostics read back
        dict(name="pd_256", kind="pd", nx=256, ny=256, L=60, M=32768, prec="f32", ragged=False, iters=10, blocks=1,
             precond=False, adaptive=False),
        # the solver in FP64 on a small ragged problem with data blocks, preconditioner and adaptive bounds
        dict(name="pd_128_f64_blocks", kind="pd", nx=128, ny=128, L=6, M=9000, prec="f64", ragged=True, iters=10,
             blocks=3, precond=True, adaptive=True),
    ]


SIDES = (64, 96, 128, 160, 192, 256, 320, 384, 512, 640, 768, 1024)   # 1, 3 or 5 times a power of two


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("phi_fwd", "phi_adj", "phi_pair", "psi_fwd", "psi_adj", "l21", "nuclear", "grad", "pd"))
    while True:
        nx = rng.choice(SIDES)
        ny = nx if rng.random() < 0.6 else rng.choice(SIDES)
        L = _log(rng, 1, 64)
        f64 = kind in ("phi_fwd", "phi_adj", "phi_pair", "psi_fwd", "psi_adj", "pd") and rng.random() < 0.2
        most = 600_000 if f64 else (4_200_000 if kind in ("pd", "grad") else 17_000_000)   # pixels of the cube
        if nx * ny * L <= most:
            break
    c = dict(kind=kind, nx=nx, ny=ny, L=L, prec="f64" if f64 else "f32")
    if kind in ("phi_fwd", "phi_adj", "phi_pair", "grad", "pd"):
        most = 60_000 if f64 else 2_000_000
        c["M"] = min(_log(rng, 300, 4 * nx * ny), max(300, most // L))
        c["ragged"] = rng.random() < 0.5
    if kind in ("phi_fwd", "phi_adj", "phi_pair"):
        c["weights"] = rng.random() < 0.3
        c["compensated"] = not f64 and rng.random() < 0.15
    if kind == "l21":
        c["dual"], c["weights"] = rng.random() < 0.5, rng.random() < 0.5
    if kind == "nuclear":
        c["dual"] = rng.random() < 0.5
    if kind == "pd":
        c["iters"] = rng.choice((1, 3, 10))
        c["blocks"] = rng.choice((1, 1, 2, 5))
        c["precond"], c["adaptive"] = rng.random() < 0.3, rng.random() < 0.3
    return c


def _levels(nx, ny):
    """Wavelet levels of an image: four, or as many as the sides allow."""
    n = 0
    while n < 4 and all(s % 2 ** (n + 1) == 0 and (s >> (n + 1) < 16 or (s >> (n + 1)) % 16 == 0) for s in (nx, ny)):
        n += 1
    return max(1, n)


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _offsets(case):
    """Visibility offsets: M per channel, or (ragged) between a quarter and all of M and one channel empty
    (a property of the case: other seeds give other data on as many visibilities)."""
    L, M = case["L"], case["M"]
    Ml = np.full(L, M, dtype=np.int64)
    if case["ragged"]:
        r = np.random.Generator(np.random.PCG64(M))
        Ml = r.integers(max(1, M // 4), M + 1, size=L)
        if L > 2:
            Ml[r.integers(1, L)] = 0
    return np.concatenate([[0], np.cumsum(Ml)]).astype(np.int64)


def _coverage(case, off, g):
    """uv in radians: N(0, (pi/4)^2) per axis at the lowest frequency, scaled by nu_l / nu_0 over one octave,
    points that would leave the band at the highest channel drawn again."""
    L = case["L"]
    fr = np.linspace(1.0, 2.0, L) if L > 1 else np.ones(1)
    n = max(1, int(np.diff(off).max()))
    lim = 0.9999 * math.pi / fr[-1]
    pool = torch.empty((0, 2), dtype=torch.float64, device="cuda")
    while pool.shape[0] < n:
        d = torch.randn((int(1.4 * n) + 64, 2), generator=g, dtype=torch.float64, device="cuda") * (math.pi / 4)
        pool = torch.cat([pool, d[d.abs().amax(dim=1) < lim]])
    uv = torch.cat([pool[:off[l + 1] - off[l]] * float(fr[l]) for l in range(L)])
    return uv.to(_real(case)).contiguous()


def _real(case):
    return torch.float32 if case["prec"] == "f32" else torch.float64


def _complex(case):
    return torch.complex64 if case["prec"] == "f32" else torch.complex128


def _sky(case, g, noise):
    """A model cube: Gaussian sources with power-law spectra on a faint background, plus noise."""
    L, ny, nx = case["L"], case["ny"], case["nx"]
    Q = 4
    u = torch.rand((Q, 5), generator=g, dtype=torch.float64, device="cuda")
    sg = 2.0 + 3.0 * u[:, 0]
    cx, cy = nx * (0.25 + 0.5 * u[:, 1]), ny * (0.25 + 0.5 * u[:, 2])
    amp, al = 0.5 + 0.5 * u[:, 3], 2.0 * u[:, 4] - 1.0
    yy = torch.arange(ny, dtype=torch.float64, device="cuda")[None, :]
    xx = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    gy = torch.exp(-(yy - cy[:, None]) ** 2 / (2 * sg[:, None] ** 2))
    gx = torch.exp(-(xx - cx[:, None]) ** 2 / (2 * sg[:, None] ** 2))
    S = (amp[:, None, None] * gy[:, :, None] * gx[:, None, :]).reshape(Q, -1)
    fr = torch.linspace(1.0, 2.0, max(L, 2), dtype=torch.float64, device="cuda")[:L]
    X = ((fr[:, None] ** -al[None, :]) @ S).reshape(L, ny, nx).to(_real(case))
    if noise:
        X += noise * torch.randn(X.shape, generator=g, dtype=_real(case), device="cuda")
    return X


def _inputs(case, seed):
    """The tensors of a case, from the seed alone (no call into the library)."""
    g = _gen(seed)
    kind, rd, cd = case["kind"], _real(case), _complex(case)
    L, ny, nx = case["L"], case["ny"], case["nx"]
    d = {}
    if "M" in case:
        d["off"] = _offsets(case)
        M = int(d["off"][-1])
        d["uv"] = _coverage(case, d["off"], g)
        if case.get("weights"):
            d["weights"] = 0.5 + torch.rand(M, generator=g, dtype=rd, device="cuda")
        if case.get("precond"):
            d["precond"] = 0.25 + torch.rand(M, generator=g, dtype=rd, device="cuda")
    else:   # prior-only calls: the plan carries a token coverage
        d["off"] = np.arange(L + 1, dtype=np.int64) * 16
        d["uv"] = (torch.rand((16 * L, 2), generator=g, dtype=torch.float64, device="cuda") - 0.5).to(rd)
    if kind in ("phi_fwd", "phi_pair", "psi_fwd"):
        d["X"] = _sky(case, g, 0.02)
    if kind in ("phi_adj", "phi_pair"):
        d["Y"] = torch.randn(M, generator=g, dtype=cd, device="cuda")
    if kind in ("psi_adj", "l21"):   # heavy-tailed coefficients whose rows differ in size
        d["A"] = torch.randn((9, L, ny, nx), generator=g, dtype=rd, device="cuda")
        d["A"] *= torch.randn((9, 1, ny, nx), generator=g, dtype=rd, device="cuda")
    if kind == "l21":
        d["thr"] = 0.5 * math.sqrt(L)
        d["w"] = torch.rand((9, ny, nx), generator=g, dtype=rd, device="cuda") if case["weights"] else None
    if kind == "nuclear":   # sources above the threshold, the noise below it
        d["X"] = _sky(case, g, 0.02)
        d["thr"] = 1.1 * 0.02 * (math.sqrt(nx * ny) + math.sqrt(L))
    if kind in ("grad", "pd"):
        truth = _sky(case, g, 0.0)
        y = _Exact(case, d).phi(truth.double())
        sigma = 1e-2 * float(torch.linalg.vector_norm(y)) / math.sqrt(max(M, 1))
        d["Y"] = (y + sigma * torch.randn(M, generator=g, dtype=torch.complex128, device="cuda")).to(cd)
        if kind == "grad":
            d["X"] = 0.7 * truth + 0.01 * torch.randn(truth.shape, generator=g, dtype=rd, device="cuda")
        else:   # equal data blocks inside each channel (an empty channel keeps empty ones)
            nb = case["blocks"]
            o = d["off"]
            b = [o[l] + (o[l + 1] - o[l]) * k // nb for l in range(L) for k in range(nb)] + [o[-1]]
            d["blk"] = np.array(b, dtype=np.int64)
            n = np.diff(d["blk"]).astype(np.float64)
            d["eps"] = torch.tensor(sigma * np.sqrt(n + 2.0 * np.sqrt(n)), dtype=torch.float64, device="cuda")
    return d


def _two_digits(v):
    return float("%.1e" % v) if v > 0 else v


def prepare(case, seed):
    d = _inputs(case, seed)
    st = {"case": case, **d}
    kind = case["kind"]
    kw = dict(levels=_levels(case["nx"], case["ny"]), prec=case["prec"])
    if kind == "pd" and case["blocks"] > 1:
        kw["blocks"] = d["blk"]
    plan = hs.Plan(case["nx"], case["ny"], d["off"], d["uv"], weights=d.get("weights"), precond=d.get("precond"),
                   compensated=case.get("compensated", False), **kw)
    st["plan"] = plan
    if kind == "pd":   # what a solve is set up with: mu from the dirty cube, the step size from the operator's norm
        mu = _two_digits(plan.estimate_mu(d["Y"])[0])
        kappa3 = _two_digits(0.95 / plan.op_norm2(iters=30, tol=1e-3))
        st["mu"], st["kappa3"] = mu, kappa3
        st["pd"] = hs.PDState(plan, d["Y"], d["eps"], kappa3=kappa3, mu=mu)
        if case["adaptive"]:
            st["pd"].set_adaptive()
    return st


def run(st):
    case, plan = st["case"], st["plan"]
    kind = case["kind"]
    if kind == "phi_fwd":
        return plan.phi_fwd(st["X"])
    if kind == "phi_adj":
        return plan.phi_adj(st["Y"])
    if kind == "phi_pair":
        return plan.phi_fwd(st["X"]), plan.phi_adj(st["Y"])
    if kind == "psi_fwd":
        return plan.psi_fwd(st["X"])
    if kind == "psi_adj":
        return plan.psi_adj(st["A"])
    if kind == "l21":
        return plan.prox_l21(st["A"], st["thr"], st["w"], dual=case["dual"])
    if kind == "nuclear":   # the prox and the singular values (FP32-accurate, as the plan's data)
        out, sv = plan.prox_nuclear(st["X"], st["thr"], dual=case["dual"])
        return out, sv.to(out.dtype)
    if kind == "grad":
        X = st["X"].detach().requires_grad_(True)
        f = hsg.objective(plan, X, st["Y"])
        (g,) = torch.autograd.grad(f, X)
        return f.detach(), g
    # pd: the iterations, then the image, beta and the residuals per data block (of the plan's precision)
    st["pd"].solve(case["iters"])
    X, beta, rho = st["pd"].get()
    return X, beta, rho.astype(np.float32 if case["prec"] == "f32" else np.float64)


# ---------------------------------------------------------------- what a pass cannot do without
def work(case):
    N, L = case["nx"] * case["ny"], case["L"]
    r = 4 if case["prec"] == "f32" else 8
    M = int(_offsets(case)[-1]) if "M" in case else 0
    K2 = 4 * N
    # one direction of the measurement operator: the cube, uv and the visibilities; a transform of a real
    # (Hermitian) K x K grid per channel and 8 x 8 complex multiply-adds per visibility
    phi_b = r * N * L + 4 * r * M + (r * M if case.get("weights") else 0)
    phi_f = L * 2.5 * K2 * math.log2(K2) / 2 + 64 * 4 * M
    # one direction of the dictionary: two separable passes of 2p-tap filters per level, p = 1 .. 8
    psi_b = 10 * r * N * L
    psi_f = L * N * 72 * 4 * sum(0.25 ** k for k in range(_levels(case["nx"], case["ny"])))
    kind = case["kind"]
    if kind in ("phi_fwd", "phi_adj"):
        b, f = phi_b, phi_f
    elif kind == "phi_pair":
        b, f = 2 * phi_b - (3 if case["weights"] else 2) * r * M, 2 * phi_f   # uv and weights once
    elif kind in ("psi_fwd", "psi_adj"):
        b, f = psi_b, psi_f
    elif kind == "l21":
        b, f = 18 * r * N * L + (9 * r * N if case["weights"] else 0), 4 * 9 * N * L
    elif kind == "nuclear":
        b, f = 2 * r * N * L, N * L * (L + 1) + 16.0 * N * L
    elif kind == "grad":
        b, f = 2 * r * N * L + 4 * r * M, 2 * (phi_f + psi_f) + 4 * 9 * N * L
    else:   # per iteration: X, X~, P and the 9 coefficient cubes read and written, v too, y and uv read
        per_b = 2 * r * N * L * (3 + 9) + 2 * 2 * r * M + 4 * r * M
        per_f = 2 * (phi_f + psi_f) + 6 * 9 * N * L + N * L * (L + 1) + 16.0 * N * L
        b, f = case["iters"] * per_b, case["iters"] * per_f
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------- 64-bit restatement
def _daubechies(p):
    """Minimum-phase Daubechies low-pass filter of 2p taps (sum sqrt 2) by spectral factorisation: the roots
    inside the unit circle of the half-band polynomial, each polished by Newton steps."""
    # P(y) = sum_k C(p-1+k, k) y^k, y = (2 - z - 1/z) / 4: one z inside the circle per root y
    c = [math.comb(p - 1 + k, k) for k in range(p)]
    h = np.array([1.0 + 0j])
    for y in (np.roots(c[::-1]) if p > 1 else []):
        for _ in range(30):
            f = sum(ck * y ** k for k, ck in enumerate(c))
            df = sum(k * ck * y ** (k - 1) for k, ck in enumerate(c) if k)
            y = y - f / df
        b = 1.0 - 2.0 * y
        z = b - np.sqrt(b * b - 1.0 + 0j)
        if abs(z) > 1.0:
            z = b + np.sqrt(b * b - 1.0 + 0j)
        h = np.convolve(h, [1.0, -z])
    for _ in range(p):
        h = np.convolve(h, [1.0, 1.0])
    h = h.real
    return h * (math.sqrt(2.0) / h.sum())


class _Exact:
    """Phi, Psi and their adjoints in FP64 from their definitions (Sec. 2.1 and 2.3), channel by channel."""

    def __init__(self, case, d):
        self.case, self.d = case, d
        self.nx, self.ny, self.L = case["nx"], case["ny"], case["L"]
        self.Kx, self.Ky = 2 * self.nx, 2 * self.ny

    def _window(self, t):
        c0 = torch.floor(t)
        cells = c0[:, None] + torch.arange(-3, 5, device="cuda", dtype=torch.float64)[None, :]
        x = t[:, None] - cells
        return cells.long(), torch.special.i0(BETA * torch.sqrt(torch.clamp(1.0 - (2.0 * x / J) ** 2, min=0.0)))

    def _scale(self, n, K):
        f = (torch.arange(n, dtype=torch.float64, device="cuda") - n // 2) / K
        s = torch.sqrt(BETA ** 2 - (math.pi * J * f) ** 2)
        return s / (J * torch.sinh(s))

    def _chunks(self, l):
        off = self.d["off"]
        for a in range(int(off[l]), int(off[l + 1]), 1 << 17):
            b = min(a + (1 << 17), int(off[l + 1]))
            uv = self.d["uv"][a:b].double()
            cx, wx = self._window(uv[:, 0] * self.Kx / (2.0 * math.pi))
            cy, wy = self._window(uv[:, 1] * self.Ky / (2.0 * math.pi))
            idx = (cy % self.Ky)[:, :, None] * self.Kx + (cx % self.Kx)[:, None, :]
            w = self.d.get("weights")
            th = 1.0 if w is None else w[a:b].double()
            yield a, b, idx, wy[:, :, None] * wx[:, None, :], th

    def phi(self, X):
        Y = torch.zeros(int(self.d["off"][-1]), dtype=torch.complex128, device="cuda")
        sc = self._scale(self.ny, self.Ky)[:, None] * self._scale(self.nx, self.Kx)[None, :]
        iy = (torch.arange(self.ny, device="cuda") - self.ny // 2) % self.Ky
        ix = (torch.arange(self.nx, device="cuda") - self.nx // 2) % self.Kx
        for l in range(self.L):
            pad = torch.zeros((self.Ky, self.Kx), dtype=torch.float64, device="cuda")
            pad[iy[:, None], ix[None, :]] = sc * X[l]
            F = torch.fft.fft2(pad).reshape(-1)
            for a, b, idx, w, th in self._chunks(l):
                Y[a:b] = th * (F[idx] * w).sum(dim=(1, 2))
        return Y

    def phi_adj(self, Y):
        X = torch.zeros((self.L, self.ny, self.nx), dtype=torch.float64, device="cuda")
        sc = self._scale(self.ny, self.Ky)[:, None] * self._scale(self.nx, self.Kx)[None, :]
        iy = (torch.arange(self.ny, device="cuda") - self.ny // 2) % self.Ky
        ix = (torch.arange(self.nx, device="cuda") - self.nx // 2) % self.Kx
        for l in range(self.L):
            G = torch.zeros((self.Ky * self.Kx, 2), dtype=torch.float64, device="cuda")
            for a, b, idx, w, th in self._chunks(l):
                v = torch.view_as_real((th * Y[a:b])[:, None, None] * w)
                G.index_add_(0, idx.reshape(-1), v.reshape(-1, 2))
            f = torch.fft.ifft2(torch.view_as_complex(G).reshape(self.Ky, self.Kx)) * (self.Kx * self.Ky)
            X[l] = sc * f.real[iy[:, None], ix[None, :]]
        return X

    def _filters(self, p):
        h = _daubechies(p)
        return h, np.array([(-1) ** j * h[2 * p - 1 - j] for j in range(2 * p)])

    @staticmethod
    def _down(x, f, dim):
        y = 0
        for j, v in enumerate(f):
            y = y + float(v) * torch.roll(x, -j, dims=dim)
        return y.index_select(dim, torch.arange(0, x.shape[dim], 2, device=x.device))

    @staticmethod
    def _up(a, f, dim):
        s = list(a.shape)
        s[dim] *= 2
        z = torch.zeros(s, dtype=a.dtype, device=a.device)
        z.index_copy_(dim, torch.arange(0, s[dim], 2, device=a.device), a)
        y = 0
        for j, v in enumerate(f):
            y = y + float(v) * torch.roll(z, j, dims=dim)
        return y

    def psi(self, X):
        A = torch.empty((9,) + tuple(X.shape), dtype=torch.float64, device="cuda")
        A[0] = X
        for p in range(1, 9):
            h, g = self._filters(p)
            A[p] = X
            m, n = self.ny, self.nx
            for _ in range(_levels(self.nx, self.ny)):
                B = A[p][:, :m, :n].clone()
                lo, hi = self._down(B, h, 2), self._down(B, g, 2)
                A[p][:, :m // 2, :n // 2] = self._down(lo, h, 1)
                A[p][:, :m // 2, n // 2:n] = self._down(hi, h, 1)
                A[p][:, m // 2:m, :n // 2] = self._down(lo, g, 1)
                A[p][:, m // 2:m, n // 2:n] = self._down(hi, g, 1)
                m, n = m // 2, n // 2
        return A / 3.0

    def psi_adj(self, A):
        X = A[0].double().clone()
        for p in range(1, 9):
            h, g = self._filters(p)
            W = A[p].double().clone()
            for k in reversed(range(_levels(self.nx, self.ny))):
                m, n = self.ny >> k, self.nx >> k
                lo = self._up(W[:, :m // 2, :n // 2], h, 1) + self._up(W[:, m // 2:m, :n // 2], g, 1)
                hi = self._up(W[:, :m // 2, n // 2:n], h, 1) + self._up(W[:, m // 2:m, n // 2:n], g, 1)
                W[:, :m, :n] = self._up(lo, h, 2) + self._up(hi, g, 2)
            X += W
        return X / 3.0


def _svt(X, thr, dual):
    """Singular values of the pixels x channels matrix and its soft threshold (or what that takes away)."""
    Z = X.reshape(X.shape[0], -1)
    lam, V = torch.linalg.eigh(Z @ Z.T)
    s = torch.sqrt(torch.clamp(lam, min=0.0))
    keep = torch.where(s > thr, thr / torch.where(s > 0, s, torch.ones_like(s)), torch.ones_like(s))
    f = keep if dual else 1.0 - keep
    return (((V * f) @ V.T) @ Z).reshape(X.shape), torch.flip(s, dims=(0,))


def exact(case, seed):
    d = _inputs(case, seed)
    e = _Exact(case, d)
    kind = case["kind"]
    if kind == "phi_fwd":
        return e.phi(d["X"].double())
    if kind == "phi_adj":
        return e.phi_adj(d["Y"].to(torch.complex128))
    if kind == "phi_pair":
        return e.phi(d["X"].double()), e.phi_adj(d["Y"].to(torch.complex128))
    if kind == "psi_fwd":
        return e.psi(d["X"].double())
    if kind == "psi_adj":
        return e.psi_adj(d["A"])
    if kind == "l21":
        A = d["A"].double()
        n = torch.sqrt((A * A).sum(dim=1, keepdim=True))
        lam = d["thr"] * (torch.ones_like(n) if d["w"] is None else d["w"].double()[:, None])
        keep = torch.where(n > lam, lam / torch.where(n > 0, n, torch.ones_like(n)), torch.ones_like(n))
        return A * (keep if case["dual"] else 1.0 - keep)
    if kind == "nuclear":
        return _svt(d["X"].double(), d["thr"], case["dual"])
    if kind == "grad":
        X, Y = d["X"].double(), d["Y"].to(torch.complex128)
        r = e.phi(X) - Y
        A = e.psi(X)
        n = torch.sqrt((A * A).sum(dim=1, keepdim=True))
        f = 0.5 * (r.real ** 2 + r.imag ** 2).sum() + n.sum()
        A /= torch.where(n > 0, n, torch.ones_like(n))
        return f, e.phi_adj(r) + e.psi_adj(A)
    return None   # pd: its step size and mu come from the library's own set-up calls
