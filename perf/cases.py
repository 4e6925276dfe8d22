"""Performance cases: what a user of the HB-UGKS library has it do, through its public entry points.

A case marches one cavity (or a batch of cavities in one handle) by a number of iterations from a given state and
reads back what a program monitors: the residuals and the conservative variables of every level; the restart case
also uploads a checkpoint and reads the harmonics and the whole state back.  Runs in single-precision storage
("fp32") hand their results on as 32-bit values, which is what that storage resolves; FP64 runs as 64-bit values.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch

from paper_2605_03479_gb300 import inputs as I

# The cavity of one case.  drive: "shear" (lid moving in its own plane), "thermal" (heated bottom wall),
# "thermal_top" (heated top wall).  mesh: "uniform", "stretched" (adjacent-cell ratio 1.1) or "refined" (0.001 of
# the height at every wall).  grid: "midpoint" or "gauss_hermite" velocities.  td: time steps per period of the
# explicit time-domain mode (0: harmonic balance).
BASE = {"kind": "march", "drive": "shear", "nx": 32, "ny": 32, "nu": 24, "nv": 24, "nh": 1, "kn": 0.1, "st": 1.0,
        "pr": 2.0 / 3.0, "amp": 0.01, "mesh": "uniform", "grid": "midpoint", "fp32": True, "implicit": False,
        "harmonic_step": False, "td": 0, "iters": 1}


def _c(name, **kw):
    return dict(BASE, name=name, **kw)


def listed():
    return [
        # the smallest use: a coarse trial cavity, marched in long calls; launches and latency
        _c("shear8_v16_nh1_fp32", nx=8, ny=8, nu=16, nv=16, amp=0.02, iters=100),
        # shear benchmark in full FP64 (BGK), the accuracy path on a modest grid
        _c("shear32_v24_nh1_fp64", pr=1.0, fp32=False, iters=10),
        # parameter sweep of the stretched shear cavity, twelve (Kn, St) pairs in one FP64 handle
        _c("sweep12_shear64_v32_nh1_fp64", kind="sweep", nx=64, ny=64, nu=32, nv=32, mesh="stretched", fp32=False,
           iters=2),
        # thermal benchmark, production precision
        _c("thermal64_v48_nh3_fp32", drive="thermal", nx=64, ny=64, nu=48, nv=48, nh=3, kn=0.5, amp=0.5, iters=10),
        # the same in FP64: the finishing iterations of a mixed-precision run
        _c("thermal64_v48_nh3_fp64", drive="thermal", nx=64, ny=64, nu=48, nv=48, nh=3, kn=0.5, amp=0.5, fp32=False,
           iters=2),
        # 48 uneven cavities iterated together in one handle
        _c("batch48_fp32", kind="batch", drive="thermal", amp=0.5, iters=2),
        # the headline: the large thermal cavity with eleven levels
        _c("thermal128_v64_nh5_fp32", drive="thermal", nx=128, ny=128, nu=64, nv=64, nh=5, kn=0.05, st=5.0, amp=0.5,
           iters=4),
        # the wall-refined shear cavity with 28-point Gauss-Hermite velocities
        _c("refined90_gh28_nh1_fp32", nx=90, ny=90, nu=28, nv=28, st=30.0, amp=0.0015, mesh="refined",
           grid="gauss_hermite", iters=10),
        # explicit time marching on the same kernels (one level, a global step), which HB is compared against
        _c("timedomain32_v24_fp32", nh=0, st=2.0, td=1235, iters=50),
        # spectral source solved at the new iterate (option for high Strouhal numbers)
        _c("implicit32_v32_nh5_fp32", drive="thermal", nu=32, nv=32, nh=5, kn=0.05, st=5.0, amp=0.5, implicit=True,
           iters=10),
        # ragged tiles, odd velocity counts with zero nodes, harmonic-mean face step
        _c("odd45x37_v31x25_nh2_fp32", drive="thermal", nx=45, ny=37, nu=31, nv=25, nh=2, kn=0.2, st=2.0, amp=0.3,
           harmonic_step=True, iters=20),
        # restart: checkpoint from the host, march, all harmonics and the checkpoint back to the host
        _c("restart32_v32_nh3_fp32", kind="restart", drive="thermal", nu=32, nv=32, nh=3, kn=0.5, amp=0.5, iters=20),
    ]


MAX_UPDATES = 70_000_000          # cell x velocity x level updates of a drawn case, per iteration


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    c = dict(BASE)
    c["kind"] = "restart" if rng.random() < 0.1 else "march"
    c["drive"] = rng.choice(["shear", "thermal", "thermal_top"])
    c["amp"] = round(rng.uniform(0.0015, 0.02) if c["drive"] == "shear" else rng.uniform(0.2, 0.5), 4)
    c["grid"] = "gauss_hermite" if rng.random() < 0.25 else "midpoint"
    c["mesh"] = rng.choice(["uniform", "uniform", "stretched", "refined"])
    c["kn"] = round(10.0 ** rng.uniform(-2.0, 1.0), 4)
    c["st"] = round(10.0 ** rng.uniform(-1.0, 1.0), 4)
    c["pr"] = 1.0 if rng.random() < 0.15 else 2.0 / 3.0
    c["fp32"] = rng.random() < 0.65
    c["harmonic_step"] = rng.random() < 0.2
    c["implicit"] = rng.random() < 0.15
    marching = rng.random() < 0.1               # explicit time marching
    c["nh"] = 0 if marching else rng.randint(1, 5)
    if marching:
        c["st"], c["implicit"], c["grid"], c["mesh"] = round(rng.uniform(2.0, 30.0), 4), False, "midpoint", "uniform"
    limit = MAX_UPDATES if c["kind"] == "march" else MAX_UPDATES // 8
    while True:
        c["nx"], c["ny"] = log_int(8, 128), log_int(8, 128)
        top = 28 if c["grid"] == "gauss_hermite" else 32 if marching else 64
        c["nu"] = rng.randint(12, top)
        c["nv"] = c["nu"] if rng.random() < 0.6 else rng.randint(12, top)
        if updates(c) <= limit:
            break
    if marching:                                # steps per period at a CFL number of 0.8 on [-4, 4]^2, or a few more
        c["td"] = math.ceil(2.0 * math.pi / c["st"] * 5.5 * (c["nx"] + c["ny"]) / 0.8 * rng.uniform(1.0, 1.3))
    cost = 1.0 if c["fp32"] else 16.0           # FP64 iterations cost more: fewer of them
    c["iters"] = max(1, min(100, int(10.0 ** rng.uniform(7.5, 8.8) / (cost * updates(c)))))
    return c


def updates(c):
    """Cell x velocity x level updates of one iteration of one cavity."""
    return c["nx"] * c["ny"] * c["nu"] * c["nv"] * (2 * c["nh"] + 1)


def work(case):
    """The state has to be read and written once per iteration; per update about 310 + 6 N_H operations (limited
    slopes 32, two reconstructions 8, two interface fluxes 110, two equilibria 60, update 32, moments 68)."""
    pair = 8 if case["fp32"] else 16            # bytes of the (h, b) pair of one update
    total = sum(k.updates_per_iteration() * (310 + 6 * k.n_harmonics) for k in _cavities(case, 0)[0])
    count = sum(k.updates_per_iteration() for k in _cavities(case, 0)[0])
    extra = 4 * 8 * count if case["kind"] == "restart" else 0       # checkpoint in and out, FP64 h and b
    return {"bytes": case["iters"] * count * 2 * pair + extra, "flops": case["iters"] * total}


# ------------------------------------------------------------------------------------------------ inputs

def _cavities(case, seed):
    """The cavities of a case and the factor each drive amplitude was scaled with (from the seed)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    if case["kind"] == "batch":
        cav = I.config4_cases()
    elif case["kind"] == "sweep":
        cav = I.config2_cases()
    else:
        kw = {"uniform": {}, "stretched": {"stretched_ratio": 1.1}, "refined": {"ds_min": 0.001}}[case["mesh"]]
        c = I.make_case(case.get("name", "drawn"), case["nx"], case["nu"], kn=case["kn"], st=case["st"], nh=case["nh"],
                        pr=case["pr"], drive=case["drive"], amp=case["amp"], precision=1 if case["fp32"] else 0,
                        ncell_y=case["ny"], nvel_y=case["nv"], vgrid=case["grid"], **kw)
        cav = [dataclasses.replace(c, face_step=int(case["harmonic_step"]), td_steps=case["td"],
                                   spectral_implicit=int(case["implicit"]))]
    out = []
    for c in cav:                               # drive amplitudes vary with the seed
        f = 0.9 + 0.2 * float(rng.random())
        out.append(dataclasses.replace(c, walls=[w[:3] + [f * x for x in w[3:]] for w in c.walls]))
    return out, rng


def _perturbed(c, rng, dev):
    """A smooth perturbation of the rest state on every level, in FP64: W (nt, ny, nx, 4) and the reduced
    Gaussians h, b (nt, ny, nx, nv, nu) of that state."""
    f64 = dict(dtype=torch.float64, device=dev)
    x = torch.tensor(0.5 * (c.xnodes[1:] + c.xnodes[:-1]), **f64)
    y = torch.tensor(0.5 * (c.ynodes[1:] + c.ynodes[:-1]), **f64)
    k = torch.arange(3, **f64)
    cx, cy = torch.cos(math.pi * k[:, None] * x), torch.cos(math.pi * k[:, None] * y)
    coef = torch.tensor(rng.uniform(-1.0, 1.0, (c.nt, 4, 3, 3)), **f64)
    f = 0.01 / 3.0 * torch.einsum("nqab,ai,bj->qnji", coef, cx, cy)
    rho, U, V, T = 1.0 + f[0], f[1], f[2], 1.0 + f[3]
    W = torch.stack([rho, rho * U, rho * V, 0.5 * rho * (U * U + V * V) + 0.75 * rho * T], -1)
    u, v = torch.tensor(c.u, **f64), torch.tensor(c.v, **f64)
    eu = torch.exp(-(u - U[..., None]) ** 2 / T[..., None])
    ev = torch.exp(-(v - V[..., None]) ** 2 / T[..., None])
    h = (rho / (math.pi * T))[..., None, None] * ev[..., :, None] * eu[..., None, :]
    return W, h, 0.5 * T[..., None, None] * h


def _start(case, seed):
    """Cavities and, where the state is small enough to hand over from the host, the initial states."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    cav, rng = _cavities(case, seed)
    if case["kind"] == "batch" or updates(case) > MAX_UPDATES:
        uniform = [(1.0 + 0.01 * float(r[0]), 0.01 * float(r[1]), 0.01 * float(r[2]), 1.0 + 0.01 * float(r[3]))
                   for r in rng.uniform(-1.0, 1.0, (len(cav), 4))]
        return cav, uniform, None
    return cav, None, [_perturbed(c, rng, dev) for c in cav]


def prepare(case, seed):
    from paper_2605_03479_gb300 import hbugks as hb
    cav, uniform, states = _start(case, seed)
    s = hb.Solver(cav)
    host = None
    if uniform is not None:                     # large grids start from a uniform state and a developed wall layer
        for k, r in enumerate(uniform):
            s.init_uniform(k, *r)
        s.iterate(8)
    elif case["kind"] == "restart":
        host = [t.cpu().numpy() for t in states[0]]
    else:
        for k, st in enumerate(states):
            s.set_state(k, *[t.cpu().numpy() for t in st])
    return {"solver": s, "cavities": cav, "iters": case["iters"], "single": case["fp32"], "checkpoint": host}


def run(state):
    s, cav, host = state["solver"], state["cavities"], state["checkpoint"]
    if host is not None:
        s.set_state(0, *host)
    _, its, res = s.iterate(state["iters"])
    out = {"iterations": its, "residual": res, "W": [s.get_W(k) for k in range(len(cav))]}
    if len(cav) > 1:
        out["W"] = np.concatenate([w.reshape(-1) for w in out["W"]])
    if host is not None:
        out["harmonics"] = np.stack([s.harmonic(0, k) for k in range(cav[0].n_harmonics + 1)])
        out["W"], out["h"], out["b"] = s.get_state(0)
    return _narrow(out) if state["single"] else out


def _narrow(v):
    """Results of a run in single-precision storage, as 32-bit values."""
    if isinstance(v, dict):
        return {k: _narrow(x) for k, x in v.items()}
    if isinstance(v, list):
        return [_narrow(x) for x in v]
    if v.dtype.kind == "c":
        return v.astype(np.complex64)
    return torch.from_numpy(v).float() if v.dtype.kind == "f" else v


# ------------------------------------------------------------------------- the same in 64 bits, plain torch

def exact(case, seed):
    cav, uniform, states = _start(case, seed)
    if uniform is not None or case["iters"] * sum(c.updates_per_iteration() for c in cav) > 1_500_000_000:
        return None
    out = {"iterations": np.array([case["iters"]] * len(cav)), "residual": [], "W": []}
    for c, st in zip(cav, states):
        ref = _Reference(c, st[0].device)
        W, h, b, res = ref.march(*st, case["iters"])
        out["residual"].append(res)
        out["W"].append(W.reshape(c.nt, c.nc, 4))
    if case["kind"] == "restart":
        out["W"], out["h"], out["b"] = (t.reshape(c.nt, c.nc, -1) for t in (W, h, b))
        f = ref.fields(h, b).reshape(c.nt, 8, c.nc)
        n = torch.arange(c.nt, dtype=torch.float64, device=f.device)
        out["harmonics"] = torch.stack([
            torch.einsum("n,nfc->fc", torch.polar(torch.full_like(n, 1.0 / c.nt), -2.0 * math.pi * k * n / c.nt),
                         f.to(torch.complex128)) for k in range(c.n_harmonics + 1)])
    elif len(cav) > 1:
        out["W"] = torch.cat([w.reshape(-1) for w in out["W"]])
    out["residual"] = torch.stack(out["residual"])
    return out


def _prim(W):
    rho = W[..., 0]
    U, V = W[..., 1] / rho, W[..., 2] / rho
    return rho, U, V, 0.75 * rho / (W[..., 3] - 0.5 * rho * (U * U + V * V))


def _coefficients(dG, tau):
    """Integrals over [0, dG] of the five weights of the integral solution."""
    x = dG / tau
    s = [torch.zeros_like(x) for _ in range(5)]
    xs, term = torch.clamp(x, max=1.0), torch.ones_like(x)
    terms = []
    for j in range(1, 25):
        term = term * xs / j
        terms.append(term)
    for j in range(24, 0, -1):
        t, sg = terms[j - 1], (1.0 if j % 2 else -1.0)
        s[3] = s[3] + sg * t
        s[4] = s[4] + sg * (j - 1) * t
        if j >= 2:
            s[0] = s[0] - sg * t
        if j >= 3:
            s[1] = s[1] + sg * (2 - j) * t
            s[2] = s[2] + sg * t
    phi, ex = -torch.expm1(-x), torch.exp(-x)
    big = [x - phi, 2.0 * phi - x - x * ex, 0.5 * x * x - x + phi, phi, x * ex - phi]
    power = [tau, tau * tau, tau * tau, tau, tau * tau]
    return [p * torch.where(x < 1.0, a, b) for p, a, b in zip(power, s, big)]


def _slope_coefficients(w, U, V, lam):
    """Coefficients of (a . psi) g whose moments per unit density are w (Maxwellian, one internal degree)."""
    e = U * U + V * V + 1.5 / lam
    r2, r3 = w[..., 1] - U * w[..., 0], w[..., 2] - V * w[..., 0]
    r4 = 2.0 * w[..., 3] - e * w[..., 0]
    a3 = (4.0 / 3.0) * lam * lam * (r4 - 2.0 * U * r2 - 2.0 * V * r3)
    a2, a1 = 2.0 * lam * r3 - V * a3, 2.0 * lam * r2 - U * a3
    return torch.stack([w[..., 0] - U * a1 - V * a2 - 0.5 * a3 * e, a1, a2, a3], -1)


class _Reference:
    """The scheme per velocity on whole arrays, FP64.  Distributions (ny, nx, nv, nu) per level; a y-normal face is
    treated as an x-normal one with both pairs of axes swapped."""

    def __init__(self, c, dev):
        self.c, self.dev = c, dev
        t = lambda a: torch.tensor(np.asarray(a, dtype=np.float64), dtype=torch.float64, device=dev)  # noqa: E731
        self.xn, self.yn, self.u, self.v = t(c.xnodes), t(c.ynodes), t(c.u), t(c.v)
        self.w = t(c.wv)[:, None] * t(c.wu)[None, :]
        a, w = c.alpha_vss, c.w_vss
        self.mu0 = c.kn * math.sqrt(math.pi) * 5.0 * (a + 1) * (a + 2) / (4.0 * a * (5 - 2 * w) * (7 - 2 * w))
        self.omega = c.st
        n = np.arange(c.nt)
        d = n[:, None] - n[None, :]
        with np.errstate(divide="ignore"):
            e = np.where(d == 0, 0.0, 0.5 * np.where(d % 2 == 0, 1.0, -1.0) / np.sin(np.pi * d / c.nt))
        self.E = t(e)

    def tau(self, rho, lam):
        return self.mu0 * (1.0 / lam) ** self.c.w_vss * 2.0 * lam / rho

    def wall(self, k, n, it):
        p, c = self.c.walls[k], self.c
        th = 2.0 * math.pi * ((it + 0.5) / c.td_steps if c.td_steps else n / c.nt)
        return [p[q] + p[3 + 2 * q] * math.cos(th) - p[4 + 2 * q] * math.sin(th) for q in range(3)]

    def steps(self, W):
        c = self.c
        if c.td_steps:
            return torch.full(W.shape[1:3], 2.0 * math.pi / (c.st * c.td_steps), dtype=torch.float64, device=self.dev)
        _, U, V, lam = _prim(W)
        cs = torch.sqrt(c.gamma / (2.0 * lam))
        dx, dy = (self.xn[1:] - self.xn[:-1])[None, :], (self.yn[1:] - self.yn[:-1])[:, None]
        nu = (torch.clamp(U.abs(), min=c.umax) + cs) / dx + (torch.clamp(V.abs(), min=c.vmax) + cs) / dy
        return c.cfl / (nu.amax(0) + self.omega * c.n_harmonics)

    @staticmethod
    def slope(f, xc):
        """van Leer slope along dimension 1, one-sided at the ends."""
        if f.shape[1] == 1:
            return torch.zeros_like(f)
        d = (f[:, 1:] - f[:, :-1]) / (xc[1:] - xc[:-1])[:, None, None]
        s1, s2 = torch.cat([d[:, :1], d], 1), torch.cat([d, d[:, -1:]], 1)
        p = s1 * s2
        return torch.where(p > 0, 2.0 * p / torch.where(p > 0, s1 + s2, torch.ones_like(p)), torch.zeros_like(p))

    @staticmethod
    def maxwell(rho, U, V, lam, un, ut):
        """Reduced Maxwellian over the grid (tangential, normal)."""
        en = torch.exp(-lam[..., None] * (un - U[..., None]) ** 2)
        et = torch.exp(-lam[..., None] * (ut - V[..., None]) ** 2)
        H = (rho * lam / math.pi)[..., None, None] * et[..., :, None] * en[..., None, :]
        return H, H * (0.5 / lam)[..., None, None]

    @staticmethod
    def moments(h, b, w, un, ut):
        """(1, u_n, u_t, |u|^2/2) moments, and the heat flux about their velocity."""
        x, y = un[None, :], ut[:, None]
        psi = torch.stack([w, w * x, w * y, 0.5 * w * (x * x + y * y)])
        M = torch.einsum("...vu,kvu->...k", h, psi)
        M[..., 3] += 0.5 * torch.einsum("...vu,vu->...", b, w)
        return M

    @staticmethod
    def heat(h, b, w, un, ut, U, V):
        x, y = un[None, :], ut[:, None]
        m = torch.stack([w, w * x, w * y, w * x * x, w * x * y, w * y * y, w * x ** 3, w * x * x * y, w * x * y * y,
                         w * y ** 3])
        A, B = torch.einsum("...vu,kvu->k...", h, m), torch.einsum("...vu,kvu->k...", b, m[:3])
        cx3 = A[6] - 3 * U * A[3] + 3 * U * U * A[1] - U ** 3 * A[0]
        cy3 = A[9] - 3 * V * A[5] + 3 * V * V * A[2] - V ** 3 * A[0]
        xyy = A[8] - 2 * V * A[4] + V * V * A[1] - U * (A[5] - 2 * V * A[2] + V * V * A[0])
        yxx = A[7] - 2 * U * A[4] + U * U * A[2] - V * (A[3] - 2 * U * A[1] + U * U * A[0])
        return 0.5 * (cx3 + xyy + B[1] - U * B[0]), 0.5 * (cy3 + yxx + B[2] - V * B[0])

    def plus(self, rho, U, V, lam, q, un, ut):
        """Maxwellian with the Shakhov correction."""
        H, B = self.maxwell(rho, U, V, lam, un, ut)
        e = lambda a: a[..., None, None]  # noqa: E731
        cx, cy = un[None, :] - e(U), ut[:, None] - e(V)
        s = e((1.0 - self.c.pr) * 4.0 * lam * lam / (5.0 * rho)) * (cx * e(q[0]) + cy * e(q[1]))
        r = 2.0 * e(lam) * (cx * cx + cy * cy)
        return H * (1.0 + s * (r - 4.0)), B * (1.0 + s * (r - 2.0))

    def face(self, f0, sn, st, left, WL, WR, dL, dR, dG, un, ut, w, wall=None, nin=0.0):
        """Micro flux rates (h, b) and macro flux rate of a set of faces: f0, sn, st pairs (h, b) of the upwinded
        reconstruction; left: weight of the low side per normal node; WL or WR None at a wall."""
        h0, b0 = f0
        e = lambda a: a[..., None, None]  # noqa: E731
        hk, bk = h0, b0
        if wall is not None:
            Uw, Vw, Tw = wall
            one = torch.ones((1, 1), dtype=torch.float64, device=self.dev)
            Hw, Bw = self.maxwell(one, Uw * one, Vw * one, one / Tw, un, ut)
            inc, ref = (un * nin < 0).double(), (un * nin > 0).double()
            den = (w * un.abs() * ref * Hw).sum((-1, -2))
            rw0 = (w * un.abs() * inc * h0).sum((-1, -2)) / den
            hk, bk = inc * h0 + ref * e(rw0) * Hw, inc * b0 + ref * e(rw0) * Bw
        W0 = self.moments(hk, bk, w, un, ut)
        rho, U, V, lam = _prim(W0)
        q = self.heat(hk, bk, w, un, ut, U, V)
        C = _coefficients(dG, self.tau(rho, lam))
        r1 = rho[..., None]
        aL = None if WL is None else _slope_coefficients((W0 - WL) / dL[..., None] / r1, U, V, lam)
        aR = None if WR is None else _slope_coefficients((WR - W0) / dR[..., None] / r1, U, V, lam)
        aL, aR = (aR if aL is None else aL), (aL if aR is None else aR)
        at = _slope_coefficients(self.moments(st[0], st[1], w, un, ut) / r1, U, V, lam)
        x, y = un[None, :], ut[:, None]

        def poly(a, k):                          # (a . psi) over xi per H (k = 1) or per B (k = 3)
            a = a[..., None, None, :]
            return a[..., 0] + a[..., 1] * x + a[..., 2] * y + 0.5 * a[..., 3] * (x * x + y * y + k * e(0.5 / lam))

        pn = [x * (left * poly(aL, k) + (1.0 - left) * poly(aR, k)) + y * poly(at, k) for k in (1.0, 3.0)]
        H, B = self.maxwell(rho, U, V, lam, un, ut)
        A = _slope_coefficients(-self.moments(pn[0] * H, pn[1] * B, w, un, ut) / r1, U, V, lam)
        Hp, Bp = self.plus(rho, U, V, lam, q, un, ut)
        C = [e(k) for k in C]
        F = [C[0] * P + C[1] * p * M + C[2] * poly(A, k) * M + C[3] * f + C[4] * (x * s + y * t)
             for P, p, M, k, f, s, t in zip((Hp, Bp), pn, (H, B), (1.0, 3.0), f0, sn, st)]
        F = [x * f / e(dG) for f in F]
        if wall is not None:
            rw = (w * inc * F[0]).sum((-1, -2)) * -nin / den
            F = [inc * f + ref * e(rw) * x * m for f, m in zip(F, (Hw, Bw))]
        return F, self.moments(F[0], F[1], w, un, ut)

    def divergence(self, h, b, sx, sy, W, dG, xn, un, ut, w, length, low, high):
        """Sum over the two x-normal faces of each cell of length x flux x outward normal: (h, b), W parts."""
        xc, hx = 0.5 * (xn[1:] + xn[:-1]), 0.5 * (xn[1:] - xn[:-1])
        hh = hx[:, None, None]
        lo = [f - s * hh for f, s in zip((h, b), sx)]        # reconstruction at the low and high face of each cell
        hi = [f + s * hh for f, s in zip((h, b), sx)]
        left = (un > 0).double() + 0.5 * (un == 0).double()
        pick = lambda L, R: [left * p[:, :-1] + (1.0 - left) * q[:, 1:] for p, q in zip(L, R)]  # noqa: E731
        parts = []
        d0 = hx.expand(W.shape[:2])
        parts.append(self.face([f[:, :1] for f in lo], [s[:, :1] for s in sx], [s[:, :1] for s in sy],
                               torch.zeros_like(left), None, W[:, :1], None, d0[:, :1], dG[:, :1], un, ut, w, low, 1.0))
        if W.shape[1] > 1:
            a, c = dG[:, :-1], dG[:, 1:]
            step = 2.0 * a * c / (a + c) if self.c.face_step else torch.minimum(a, c)
            parts.append(self.face(pick(hi, lo), pick(sx, sx), pick(sy, sy), left, W[:, :-1], W[:, 1:], d0[:, :-1],
                                   d0[:, 1:], step, un, ut, w))
        parts.append(self.face([f[:, -1:] for f in hi], [s[:, -1:] for s in sx], [s[:, -1:] for s in sy],
                               torch.ones_like(left), W[:, -1:], None, d0[:, -1:], None, dG[:, -1:], un, ut, w, high,
                               -1.0))
        Fh, Fb = (torch.cat([p[0][k] for p in parts], 1) for k in range(2))
        FW = torch.cat([p[1] for p in parts], 1)
        ln = length[:, None]
        return (ln[..., None, None] * (Fh[:, 1:] - Fh[:, :-1]), ln[..., None, None] * (Fb[:, 1:] - Fb[:, :-1]),
                ln[..., None] * (FW[:, 1:] - FW[:, :-1]))

    def march(self, W, h, b, iters):
        c, u, v, w = self.c, self.u, self.v, self.w
        xc, yc = 0.5 * (self.xn[1:] + self.xn[:-1]), 0.5 * (self.yn[1:] + self.yn[:-1])
        dx, dy = self.xn[1:] - self.xn[:-1], self.yn[1:] - self.yn[:-1]
        area = dy[:, None] * dx[None, :]
        tr = lambda f: f.permute(1, 0, 3, 2)  # noqa: E731
        swap = [0, 2, 1, 3]
        for it in range(iters):
            dG = self.steps(W)
            div = []
            for n in range(c.nt):
                wl = [self.wall(k, n, it) for k in range(4)]
                turned = [[x[1], x[0], x[2]] for x in wl]
                sx = [self.slope(f[n], xc) for f in (h, b)]
                sy = [tr(self.slope(tr(f[n]), yc)) for f in (h, b)]
                p = self.divergence(h[n], b[n], sx, sy, W[n], dG, self.xn, u, v, w, dy, wl[3], wl[1])
                q = self.divergence(tr(h[n]), tr(b[n]), [tr(s) for s in sy], [tr(s) for s in sx],
                                    W[n].transpose(0, 1)[..., swap], dG.T, self.yn, v, u, w.T, dx, turned[0],
                                    turned[2])
                div.append((p[0] + tr(q[0]), p[1] + tr(q[1]), p[2] + q[2].transpose(0, 1)[..., swap]))
            source = (lambda f: torch.zeros_like(f)) if c.spectral_implicit else (
                lambda f: torch.tensordot(self.E, f, dims=([1], [0])))
            Wn = W - dG[..., None] * (torch.stack([d[2] for d in div]) / area[..., None] + self.omega * source(W))
            eye = torch.eye(c.nt, dtype=torch.float64, device=self.dev)
            rot = (dG * self.omega)[..., None, None] * self.E             # (ny, nx, nt, nt)
            if c.spectral_implicit:
                Wn = torch.linalg.solve(eye + rot, Wn.permute(1, 2, 0, 3)).permute(2, 0, 1, 3)
            spec = [source(f) for f in (h, b)]
            new, D = ([], []), []
            for n in range(c.nt):
                p0, p1 = _prim(W[n]), _prim(Wn[n])
                q = self.heat(h[n], b[n], w, u, v, p0[1], p0[2])
                e = lambda a: a[..., None, None]  # noqa: E731
                k0, k1 = e(0.5 * dG / self.tau(p0[0], p0[3])), e(0.5 * dG / self.tau(p1[0], p1[3]))
                e0, e1 = self.plus(*p0, q, u, v), self.plus(*p1, q, u, v)
                D.append(1.0 + k1)
                for g, f, dv, sp, f0, f1 in zip(new, (h, b), div[n], spec, e0, e1):
                    g.append((f[n] - e(dG / area) * dv - e(dG * self.omega) * sp[n] + k1 * f1 + k0 * (f0 - f[n]))
                             / (1.0 if c.spectral_implicit else D[n]))
            hn, bn = torch.stack(new[0]), torch.stack(new[1])
            if c.spectral_implicit:
                inv = torch.linalg.inv(torch.diag_embed(torch.stack([d[..., 0, 0] for d in D], -1)) + rot)
                hn, bn = (torch.einsum("jinm,mjivu->njivu", inv, f) for f in (hn, bn))
            res = torch.sqrt(((Wn[0] - W[0]) ** 2).mean((0, 1)))
            W, h, b = Wn, hn, bn
        return W, h, b, res

    def fields(self, h, b):
        """rho, U, V, T, tau_xy, q_x, q_y, p from the moments of h and b."""
        x, y = self.u[None, :], self.v[:, None]
        rho, U, V, lam = _prim(self.moments(h, b, self.w, self.u, self.v))
        qx, qy = self.heat(h, b, self.w, self.u, self.v, U, V)
        xy = torch.einsum("...vu,vu->...", h, self.w * x * y) - rho * U * V
        return torch.stack([rho, U, V, 1.0 / lam, xy, qx, qy, rho / (2.0 * lam)], 1)
