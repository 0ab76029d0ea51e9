"""Workloads of this framework, through its public entry points, for timing.

Every case is something a user of the T-REXI step runs: single states, ensembles, long
integrations, gradients, ragged batches, and the transforms by themselves, in the arithmetic
options the plans offer.  ``exact`` is the same result from plain numpy and torch in 64 bits:
the REXI symbol of the operator by a Chebyshev expansion and dense Legendre sums, written here
from the equations and sharing nothing with the package.
"""
import functools
import math

import numpy as np
import torch

A_EARTH, OMEGA, GRAVITY, DEPTH = 6.37122e6, 7.292e-5, 9.80616, 1.0e4
PHIBAR = GRAVITY * DEPTH
WIDTH, TERMS, MU = 0.2, 11, -4.53  # h, Gaussian terms per side, and their common real part


# ---- poles -------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def poles(M):
    """(alpha, beta) of T-REXI for M Gaussian basis functions per side, renormalised at x = 0.
    A least-squares fit of the Gaussian by 2 * TERMS + 1 simple fractions, as the method has it."""
    y = np.linspace(-60.0, 60.0, 6001)
    l = np.arange(-TERMS, TERMS + 1)
    frac = 1.0 / (1j * y[:, None] + MU + 1j * l[None, :])
    c = np.linalg.lstsq(np.hstack([frac.real, -frac.imag]), np.exp(-y * y / 4) / np.sqrt(4 * np.pi), rcond=None)[0]
    a = c[: l.size] + 1j * c[l.size:]
    a = 0.5 * (a + np.conj(a[::-1]))
    J = M + TERMS
    m = np.arange(-M, M + 1)
    beta = np.zeros(2 * J + 1, dtype=complex)
    for i, li in enumerate(l):
        beta[li + m + J] += WIDTH * math.exp(WIDTH * WIDTH) * np.cos(m * WIDTH) * a[i]
    alpha = WIDTH * (MU + 1j * np.arange(-J, J + 1))
    return alpha, beta / np.sum(beta / alpha)


def npoles(M):
    return 2 * (M + TERMS) + 1


# ---- spectral states -----------------------------------------------------------------------
def nspec(N):
    return (N + 1) * (N + 2) // 2


@functools.lru_cache(maxsize=8)
def degrees(N):
    """(n, m) of every coefficient, zonal orders one after the other."""
    m = np.concatenate([np.full(N - k + 1, k) for k in range(N + 1)])
    n = np.concatenate([np.arange(k, N + 1) for k in range(N + 1)])
    return n, m


def spectra(N, B, seed, device="cuda"):
    """[B, 3, nspec] (Phi, zeta, delta): complex normal coefficients falling as n^-3, a height
    perturbation of 50 m and winds of 5 m/s, real at m = 0."""
    g = torch.Generator(device=device).manual_seed(1000 + int(seed))
    n, m = (torch.from_numpy(v).to(device) for v in degrees(N))
    amp = torch.where(n > 0, n.clamp(min=1).double() ** -3.0, 0.0)
    z = torch.randn(B, 3, n.numel(), 2, dtype=torch.float64, device=device, generator=g)
    z[..., 1] *= (m > 0)
    S = torch.view_as_complex(z) * amp
    mult = torch.where(m > 0, 1.0, 0.5)
    lap = torch.where(n > 0, A_EARTH ** 2 / (n * (n + 1)).clamp(min=1).double(), 0.0)
    power = (mult * S.abs() ** 2)
    S[:, 0] *= (GRAVITY * 50.0 / power[:, 0].sum(-1).sqrt())[:, None]
    S[:, 1:] *= (5.0 * math.sqrt(2.0) / (power[:, 1:] * lap).sum((-1, -2)).sqrt())[:, None, None]
    return S


# ---- the same in plain 64-bit torch ------------------------------------------------------------
@functools.lru_cache(maxsize=1)
def gauss(nlat):
    """Gauss-Legendre latitudes (descending sines) and weights."""
    x = np.cos(np.pi * (np.arange(nlat) + np.longdouble(0.75)) / (nlat + np.longdouble(0.5)))
    for _ in range(6):
        p0, p1 = np.ones_like(x), x.copy()
        for k in range(2, nlat + 1):
            p0, p1 = p1, ((2 * k - 1) * x * p1 - (k - 1) * p0) / k
        dp = nlat * (x * p1 - p0) / (x * x - 1)
        x = x - p1 / dp
    return x.astype(np.float64), (2 / ((1 - x * x) * dp * dp)).astype(np.float64)


def eps(n, m):
    return torch.where(n > m, ((n * n - m * m).clamp(min=0) / (4 * n * n - 1)).sqrt(), 0.0)


class Sphere:
    """Dense states X[..., m, n] (n = 0..N) and the operator, analysis and synthesis on them."""

    def __init__(self, N, nlat=None, nlon=None, device="cuda"):
        self.N, self.nlat, self.nlon = N, nlat, nlon
        d = dict(dtype=torch.float64, device=device)
        m, n = torch.arange(N + 1, **d)[:, None], torch.arange(N + 2, **d)[None, :]
        self.m, self.n, self.e = m, n, eps(n, m)
        nn, pos = n[:, :N + 1].clamp(min=1), (n[:, :N + 1] >= m) & (n[:, :N + 1] > 0)
        e0, e1 = self.e[:, :N + 1], self.e[:, 1:]
        self.sigma = torch.where(pos, 2 * OMEGA * m / (nn * (nn + 1)), 0.0)
        self.c = torch.where(pos & (nn - 1 >= m.clamp(min=1)), 2 * OMEGA * e0 * (nn + 1) / nn, 0.0)
        self.d = torch.where(pos & (nn < N), 2 * OMEGA * e1 * nn / (nn + 1), 0.0)
        self.G = torch.where(pos, nn * (nn + 1) / A_EARTH ** 2, 0.0)
        self.pos = pos
        dn, dm = degrees(N)
        self.at = torch.from_numpy(dm * (N + 1) + dn).to(device)

    def unpack(self, S):
        X = torch.zeros(S.shape[:-1] + ((self.N + 1) ** 2,), dtype=S.dtype, device=S.device)
        X = X.index_copy(-1, self.at, S).reshape(S.shape[:-1] + (self.N + 1, self.N + 1))
        return torch.cat([X[..., :1, :, :], X[..., 1:, :, :] * self.pos], dim=-3)

    def pack(self, X):
        return X.reshape(X.shape[:-2] + (-1,))[..., self.at]

    def slope(self, X):
        """L X."""
        P, Z, D = X[..., 0, :, :], X[..., 1, :, :], X[..., 2, :, :]
        lo, hi = (lambda v: torch.roll(v, 1, -1)), (lambda v: torch.roll(v, -1, -1))
        return torch.stack([-PHIBAR * D * self.pos,
                            1j * self.sigma * Z - self.c * lo(D) - self.d * hi(D),
                            1j * self.sigma * D + self.c * lo(Z) + self.d * hi(Z) + self.G * P], dim=-3)

    def rexi(self, X, M, tau, steps=1):
        """(sum_k beta_k (alpha_k + tau L)^-1)^steps X, from the symbol's Chebyshev series."""
        top = tau * (2 * OMEGA + math.sqrt(PHIBAR * self.N * (self.N + 1)) / A_EARTH)
        coef = symbol(M, top, steps)
        back = lambda v: self.slope(v) * (-1j * tau / top)  # noqa: E731
        t0, t1 = X, back(X)
        out = coef[0] * t0 + coef[1] * t1
        for k in range(2, len(coef)):
            t0, t1 = t1, 2 * back(t1) - t0
            out = out + coef[k] * t1
        return torch.cat([out[..., :1, :].real.to(out.dtype), out[..., 1:, :]], dim=-2)

    def legendre(self):
        """Pbar[m, lat, n], n = 0..N+1, and the weights; kept for the last sphere only."""
        return tables(self.N, self.nlat)

    def gradient_sum(self, psi):
        """Coefficients (n = 0..N+1) whose Legendre sum is that of (1 - mu^2) dP/dmu over psi."""
        out = torch.zeros(psi.shape[:-1] + (self.N + 2,), dtype=psi.dtype, device=psi.device)
        low = torch.nn.functional.pad(psi[..., 1:] * (self.n[:, 2:self.N + 2]) * self.e[:, 1:self.N + 1], (0, 2))
        up = torch.nn.functional.pad(psi * -self.n[:, :self.N + 1] * self.e[:, 1:], (1, 0))
        return out + low + up

    def synthesise(self, S):
        """[B, 3, nspec] -> (h', u, v) on the grid."""
        P, _, mu = self.legendre()
        X = self.unpack(S)
        inv = torch.where(self.n[:, :self.N + 1] > 0, -A_EARTH / (self.n * (self.n + 1)).clamp(min=1)[:, :self.N + 1], 0.0)
        psi, chi = X[..., 1, :, :] * inv, X[..., 2, :, :] * inv
        pad = lambda v: torch.nn.functional.pad(v, (0, 1))  # noqa: E731
        cols = torch.stack([pad(X[..., 0, :, :]) / GRAVITY, 1j * self.m * pad(chi) - self.gradient_sum(psi),
                            1j * self.m * pad(psi) + self.gradient_sum(chi)], dim=1)
        B = S.shape[0]
        r = torch.view_as_real(cols.reshape(B * 3, self.N + 1, self.N + 2)).permute(1, 2, 0, 3).reshape(self.N + 1, self.N + 2, -1)
        F = torch.bmm(P, r).reshape(self.N + 1, self.nlat, B, 3, 2).permute(2, 3, 1, 0, 4).contiguous()
        F = torch.view_as_complex(F)
        F = torch.nn.functional.pad(F, (0, self.nlon // 2 + 1 - F.shape[-1]))
        x = torch.fft.irfft(F * self.nlon, n=self.nlon, dim=-1)
        scale = torch.stack([torch.ones_like(mu), (1 - mu * mu).rsqrt(), (1 - mu * mu).rsqrt()])
        return x * scale[None, :, :, None]

    def analyse(self, x):
        """(h', u, v) on the grid -> [B, 3, nspec]."""
        P, w, mu = self.legendre()
        B = x.shape[0]
        cos = (1 - mu * mu).sqrt()
        scale = torch.stack([GRAVITY * w, w / (A_EARTH * cos), w / (A_EARTH * cos)])
        F = torch.fft.rfft(x * scale[None, :, :, None], dim=-1)[..., :self.N + 1] / self.nlon
        r = torch.view_as_real(F).permute(3, 2, 0, 1, 4).reshape(self.N + 1, self.nlat, -1)
        C = torch.bmm(P.transpose(1, 2), r).reshape(self.N + 1, self.N + 2, B, 3, 2).permute(2, 3, 0, 1, 4).contiguous()
        C = torch.view_as_complex(C)
        n, e, N = self.n, self.e, self.N

        def grad(v):
            return -n[:, :N + 1] * e[:, 1:] * v[..., 1:] + (n[:, :N + 1] + 1) * e[:, :N + 1] * torch.roll(v, 1, -1)[..., :N + 1]

        U, V = C[:, 1], C[:, 2]
        X = torch.stack([C[:, 0, :, :N + 1], 1j * self.m * V[..., :N + 1] + grad(U), 1j * self.m * U[..., :N + 1] - grad(V)], dim=1)
        S = self.pack(X)
        keep = torch.ones_like(S.real)
        keep[:, 1:, 0] = 0
        return S * keep


@functools.lru_cache(maxsize=1)
def tables(N, nlat):
    mu, w = (torch.from_numpy(v).cuda() for v in gauss(nlat))
    P = torch.zeros(N + 1, nlat, N + 2, dtype=torch.float64, device="cuda")
    m = torch.arange(N + 1, dtype=torch.float64, device="cuda")
    one = torch.full_like(mu, 1 / math.sqrt(2.0))
    before = now = torch.zeros(N + 1, nlat, dtype=torch.float64, device="cuda")
    for n in range(N + 2):
        t = torch.full((1,), float(n), dtype=torch.float64, device="cuda")
        e0, e1 = eps(t, m), eps(t - 1, m)
        new = torch.where((m < n)[:, None], (mu * now - e1[:, None] * before) / e0.clamp(min=1e-300)[:, None], 0.0)
        if n <= N:
            new[n] = one
            one = one * math.sqrt((2 * n + 3) / (2 * n + 2)) * (1 - mu * mu).sqrt()
        P[:, :, n] = new
        before, now = now, new
    return P, w, mu


@functools.lru_cache(maxsize=4)
def symbol(M, top, steps):
    """Chebyshev coefficients over [-top, top] of (sum_k beta_k / (alpha_k + i x))^steps."""
    al, be = poles(M)
    K = 256
    while K < 44 * top + 1200:
        K *= 2
    x = np.cos(np.pi * (np.arange(K) + 0.5) / K) * top
    re, im = np.zeros(K, dtype=np.longdouble), np.zeros(K, dtype=np.longdouble)
    for a, b in zip(al, be):  # b / (a + i x)
        y = x + np.longdouble(a.imag)
        q = 1 / (np.longdouble(a.real) ** 2 + y * y)
        re += (b.real * np.longdouble(a.real) + b.imag * y) * q
        im += (b.imag * np.longdouble(a.real) - b.real * y) * q
    f = (re.astype(float) + 1j * im.astype(float)) ** steps
    k = np.arange(K)
    c = np.fft.fft(np.concatenate([f, f[::-1]]))[:K] * np.exp(-0.5j * np.pi * k / K) / K
    c[0] *= 0.5
    big = np.nonzero(np.abs(c) > 3e-17 * np.abs(c).max())[0]
    return [complex(v) for v in c[: max(2, big[-1] + 1)]]


def grid_of(N):
    nlon = 3 * N + 3
    while True:
        k = nlon
        for q in (2, 3, 5):
            while k % q == 0:
                k //= q
        if k == 1 and nlon % 4 == 0:
            return nlon // 2, nlon
        nlon += 1


# ---- cases -----------------------------------------------------------------------------------
def listed():
    return [
        # the paper's validation run: one T63 state, where latency and launches count
        dict(name="t63_b1", kind="step", N=63, M=128, tau=3600.0, B=1, layout="grid", precision="fp64"),
        # a small study at an odd truncation, spectral states in and out, a few members
        dict(name="t85_b5", kind="step", N=85, M=96, tau=1800.0, B=5, layout="spectral", precision="fp64"),
        # a forecast of one state: many steps in one call (the Gaussian-bump runs)
        dict(name="t128_run", kind="integrate", N=128, M=512, tau=800.0, B=1, steps=20, layout="spectral", precision="fp64"),
        # an ensemble of many medium states in the mixed form
        dict(name="t127_b64", kind="step", N=127, M=256, tau=7200.0, B=64, layout="grid", precision="mixed"),
        # the headline batch, mixed transforms and binary64 solves
        dict(name="t341_b16", kind="step", N=341, M=256, tau=1200.0, B=16, layout="grid", precision="mixed"),
        # the same with every transform in binary64
        dict(name="t341_b16_fp64", kind="step", N=341, M=256, tau=1200.0, B=16, layout="grid", precision="fp64"),
        # a 4D-Var gradient: an eight-step rollout, checkpointed, and its backward pass
        dict(name="t170_gradient", kind="gradient", N=170, M=256, tau=3600.0, B=1, steps=8, layout="grid", precision="fp64"),
        # the same direction for an ensemble: one adjoint step of spectral states
        dict(name="t170_b16_adjoint", kind="adjoint", N=170, M=256, tau=3600.0, B=16, layout="spectral", precision="fp64"),
        # forty-eight states of mixed truncations and pole counts in one call
        dict(name="ragged_48", kind="ragged", states=48, largest=341, pick=1002),
        # one high-resolution state
        dict(name="t639_b1", kind="step", N=639, M=256, tau=7200.0, B=1, layout="grid", precision="mixed"),
        # analysis and synthesis by themselves (reading fields in, writing them out)
        dict(name="t255_transforms", kind="transforms", N=255, M=16, tau=1200.0, B=8, layout="grid", precision="fp64"),
        # the float-float solve option on an ensemble
        dict(name="t170_b12_ff", kind="step", N=170, M=256, tau=3600.0, B=12, layout="grid", precision="mixed", arith="fp32x2"),
    ]


KINDS = ["step"] * 5 + ["integrate", "gradient", "adjoint", "adjoint", "ragged", "transforms"]


def draw(rng):
    kind = rng.choice(KINDS)
    if kind == "ragged":
        return dict(kind=kind, states=rng.randint(3, 48), largest=rng.choice([127, 170, 255, 341]), pick=rng.randint(0, 10 ** 6))
    while True:
        c = dict(kind=kind, N=int(round(math.exp(rng.uniform(math.log(21), math.log(400))))),
                 M=int(round(math.exp(rng.uniform(math.log(32), math.log(512))))),
                 tau=rng.choice([600.0, 1200.0, 1800.0, 3600.0, 7200.0]), B=int(round(math.exp(rng.uniform(0.0, math.log(64))))),
                 layout=rng.choice(["grid", "spectral"]), precision=rng.choice(["fp64", "fp64", "mixed"]))
        if kind in ("integrate", "gradient"):
            c["steps"] = rng.randint(2, 12)
            c["B"] = min(c["B"], 8)
        if kind == "gradient":
            c["layout"] = "grid"
        if kind == "transforms":
            c["M"], c["layout"] = 16, "grid"
        if c["layout"] == "spectral":
            c["precision"] = "fp64"  # the mixed form is that of the transforms
        if kind == "step" and rng.random() < 0.15:
            c["arith"] = "fp32x2"
        if c["B"] * npoles(c["M"]) * nspec(c["N"]) * c.get("steps", 1) * (2 if kind == "gradient" else 1) <= 16 * npoles(256) * nspec(341) * 0.8:
            return c


def members(case):
    """(N, M) of every state of a ragged batch."""
    r = np.random.default_rng(case["pick"])
    allowed = [N for N in (63, 127, 170, 255, 341) if N <= case["largest"]]
    return [(int(r.choice(allowed)), int(r.choice([128, 256]))) for _ in range(case["states"])]


def grids(case):
    return {63: (96, 192), 127: (192, 384), 128: (192, 384), 170: (256, 512), 255: (384, 768), 341: (512, 1024),
            639: (960, 1920)}.get(case["N"]) or grid_of(case["N"])


def fields(case, seed):
    """The inputs of a case: spectral states, or grid fields synthesised from them."""
    S = spectra(case["N"], case["B"], seed)
    if case["layout"] == "spectral":
        return S
    return Sphere(case["N"], *grids(case)).synthesise(S)


def prepare(case, seed):
    from paper_1812_03431_gb300 import rexi
    if case["kind"] == "ragged":
        who = members(case)
        kinds = sorted(set(who))
        plans = []
        for N, M in kinds:
            al, be = poles(M)
            plans.append(rexi.Plan(N, *grids(dict(N=N)), tau=1200.0, max_batch=who.count((N, M)), layout="spectral", alpha=al, beta=be))
        states = [spectra(N, 1, 100 * seed + i)[0] for i, (N, _) in enumerate(who)]
        return dict(case=case, plans=plans, ragged=rexi.Ragged(plans, len(who)), plan_of=[kinds.index(w) for w in who], x=states)
    al, be = poles(case["M"])
    plan = rexi.Plan(case["N"], *grids(case), tau=case["tau"], max_batch=case["B"], layout=case["layout"], precision=case["precision"],
                     alpha=al, beta=be, solve_arith=case.get("arith", "fp64"))
    s = dict(case=case, plan=plan, x=fields(case, seed))
    if case["kind"] == "gradient":
        s["y"] = fields(case, seed + 7919)
    if case["kind"] == "transforms":
        s["spec"] = spectra(case["N"], case["B"], seed + 7919)
    return s


def run(state):
    from paper_1812_03431_gb300 import autograd
    case, x, kind = state["case"], state["x"], state["case"]["kind"]
    if kind == "ragged":
        return state["ragged"].step(x, [torch.empty_like(v) for v in x], state["plan_of"])
    plan = state["plan"]
    if kind == "step":
        return plan.step(x)
    if kind == "integrate":
        return plan.integrate(x, case["steps"])
    if kind == "adjoint":
        return plan.step_adjoint(x)
    if kind == "transforms":
        return [plan.analyze(x), plan.synthesize(state["spec"])]
    x0 = x.detach().requires_grad_(True)
    u = autograd.rollout(plan, x0, case["steps"], checkpoint_every=2)
    (grad,) = torch.autograd.grad(((u - state["y"]) ** 2).sum(), x0)
    return [u.detach(), grad]


def work(case):
    """States in and out once; the banded solves at nine complex multiply-adds per state, pole and
    row (a factored tridiagonal system, three right-hand-side couplings, four weighted sums); the
    Legendre contractions at ten multiply-adds per state, coefficient and latitude pair, and the
    longitude transforms."""
    if case["kind"] == "ragged":
        parts = [dict(kind="step", N=N, M=M, B=1, layout="spectral") for N, M in members(case)]
        each = [work(p) for p in parts]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    N, B, kind = case["N"], case["B"], case["kind"]
    nlat, nlon = grids(case)
    solve = 72.0 * B * npoles(case["M"]) * (nspec(N) - 1)
    legendre = 2 * 10.0 * B * nspec(N) * (nlat // 2)
    fft = B * 3 * nlat * 2.5 * nlon * math.log2(nlon)
    spec, grid = 48.0 * B * nspec(N), 24.0 * B * nlat * nlon
    n = case.get("steps", 1)
    if kind == "transforms":
        return {"bytes": 2 * (spec + grid), "flops": 2 * (legendre + fft)}
    if kind == "gradient":
        return {"bytes": 4 * grid, "flops": 2 * n * (solve + 2 * (legendre + fft))}
    if case["layout"] == "spectral":
        return {"bytes": 2 * spec, "flops": n * solve}
    return {"bytes": 2 * grid, "flops": n * solve + 2 * (legendre + fft)}


def exact(case, seed):
    if case["kind"] == "ragged":
        outs = []
        for i, (N, M) in enumerate(members(case)):
            if N > 170:  # the smaller members stand for the others, which would take longer
                outs.append(None)
                continue
            sp = Sphere(N)
            outs.append(sp.pack(sp.rexi(sp.unpack(spectra(N, 1, 100 * seed + i)), M, 1200.0))[0])
        return outs
    sp = Sphere(case["N"], *grids(case))
    x, kind = fields(case, seed), case["kind"]
    if kind == "transforms":
        return [sp.analyse(x), sp.synthesise(spectra(case["N"], case["B"], seed + 7919))]

    def steps(v, n):
        S = v if case["layout"] == "spectral" else sp.analyse(v)
        S = sp.pack(sp.rexi(sp.unpack(S), case["M"], case["tau"], n))
        return S if case["layout"] == "spectral" else sp.synthesise(S)

    if kind in ("step", "integrate"):
        return steps(x, case.get("steps", 1))
    if kind == "adjoint":
        x0 = torch.zeros_like(x).requires_grad_(True)
        (grad,) = torch.autograd.grad(steps(x0, 1), x0, grad_outputs=x)
        return grad
    x0 = x.detach().requires_grad_(True)
    u = steps(x0, case["steps"])
    (grad,) = torch.autograd.grad(((u - fields(case, seed + 7919)) ** 2).sum(), x0)
    return [u.detach(), grad]
