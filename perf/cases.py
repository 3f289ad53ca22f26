"""Workloads that the performance of this framework is measured on.

Each case is one step of a user's program through the Python API: a Monte
Carlo sweep with its measurements, a gradient step, time-origin averaged
G(tau), the Green functions of given fields, or the analysis of measured
G_k(tau).  `listed()` names them, `draw()` gives more of the same ranges,
`prepare()` builds what such a program holds before the call, `run()` is one
step, `work()` what a step cannot do without, and `exact()` the same results
in plain numpy FP64.

A case of kind "sweep", "grad", "origins" or "green" describes its groups of
chains by a text, one group per semicolon:
    "Lx x Ly, U, beta, dtau, chains, stab_interval, delay_k"
"""
import math

import numpy as np
import torch

import paper_1504_05090_gb300 as pkg

T_HOP = 0.25


# ---------------------------------------------------------------------------
# The cases.
# ---------------------------------------------------------------------------
def _g(Lx, Ly, U, beta, dtau, chains, ns, k):
    return "%dx%d, %g, %g, %g, %d, %d, %d" % (Lx, Ly, U, beta, dtau, chains, ns, k)


def listed():
    u, b, d = (1.0, 2.0, 3.0), (10.0, 15.0, 20.0), (0.2, 0.125, 0.1)
    uneven = "; ".join(_g(s, s, u[i % 3], b[i % 3], d[i % 3], 32, 10, 16)
                       for i, s in enumerate((6, 8, 10, 12, 14, 16)))
    return [
        # one chain on the smallest production cluster: every launch is tiny
        dict(name="sweep_4x4_1ch_fp64", kind="sweep", precision="fp64", gtau=False,
             groups=_g(4, 4, 1.0, 10.0, 0.25, 1, 10, 16)),
        # a handful of chains on an elongated cluster whose site count fills no warp
        dict(name="sweep_10x6_7ch_fp64", kind="sweep", precision="fp64", gtau=True,
             groups=_g(10, 6, 3.0, 10.0, 0.1, 7, 12, 16)),
        # the three time steps of one dtau -> 0 extrapolation, 256 chains each, in one context
        dict(name="sweep_8x8_3x256ch_df32", kind="sweep", precision="df32", gtau=True,
             groups="; ".join(_g(8, 8, 2.0, 20.0, dt, 256, 8, 16) for dt in (0.4, 0.2, 0.1))),
        # single precision with the short stabilisation interval that it needs
        dict(name="sweep_8x8_32ch_fp32", kind="sweep", precision="fp32", gtau=False,
             groups=_g(8, 8, 2.0, 10.0, 0.125, 32, 2, 16)),
        # the production sweep on the largest cluster, float-pair working precision
        dict(name="sweep_16x16_64ch_df32", kind="sweep", precision="df32", gtau=True,
             groups=_g(16, 16, 2.0, 20.0, 0.125, 64, 10, 32)),
        # the same cluster in plain FP64, half as many chains at half the beta
        dict(name="sweep_16x16_32ch_fp64", kind="sweep", precision="fp64", gtau=True,
             groups=_g(16, 16, 2.0, 10.0, 0.125, 32, 10, 32)),
        # two chains on the largest cluster: warm-up and test runs
        dict(name="sweep_16x16_2ch_df32", kind="sweep", precision="df32", gtau=False,
             groups=_g(16, 16, 2.0, 10.0, 0.125, 2, 10, 32)),
        # six cluster sizes in one context, as a finite-size study runs them
        dict(name="sweep_uneven_6x32ch_df32", kind="sweep", precision="df32", gtau=False,
             groups=uneven),
        # sweep and gradient of log W, 512 chains
        dict(name="grad_8x8_512ch_fp64", kind="grad", precision="fp64",
             groups=_g(8, 8, 2.0, 10.0, 0.125, 512, 10, 16)),
        # G(tau) averaged over four time origins on a rectangular cluster
        dict(name="origins_14x10_8ch_fp64", kind="origins", precision="fp64", origins=4,
             groups=_g(14, 10, 2.0, 5.0, 0.125, 8, 10, 16)),
        # stabilised Green functions of stored fields (reweighting, restart)
        dict(name="green_12x12_16ch_df32", kind="green", precision="df32",
             groups=_g(12, 12, 2.0, 20.0, 0.2, 16, 6, 16)),
        # dtau -> 0 extrapolation and self-energy of three measured runs, on the device
        dict(name="analysis_8x8_256ch", kind="analysis", Lx=8, Ly=8, beta=20.0, slices="50, 100, 200",
             chains=256, fine=400, freqs=200),
    ]


def _cost(groups, gtau):
    """Rough device seconds of a sweep, to keep drawn cases below the largest listed one."""
    s = 0.0
    for g in groups:
        N, L, C = g.N, g.L, g.n_chains
        s += L * N * 1.3e-6 + C * L * N ** 3 * (1.5e-12 + 8e-12 / g.stab_interval)
        s += math.ceil(L / g.stab_interval) * N * 8e-6 * (2 if gtau else 1)
    return s


def draw(rng):
    kind = rng.choice(("sweep",) * 7 + ("grad", "origins", "green", "analysis", "analysis"))
    if kind == "analysis":
        Lx, Ly = rng.choice((2, 4, 6, 8, 10, 12)), rng.choice((2, 4, 6, 8, 10, 12))
        beta = rng.choice((5.0, 10.0, 20.0))
        ls = sorted(rng.sample(range(12, 201), rng.randint(1, 4)))
        chains = min(int(round(2 ** rng.uniform(0, 9))), 40_000_000 // (8 * Lx * Ly * sum(ls)) + 1)
        return dict(kind=kind, Lx=Lx, Ly=Ly, beta=beta, slices=", ".join(map(str, ls)), chains=chains,
                    fine=rng.randint(60, 400), freqs=rng.randint(20, 200))
    while True:
        prec = "fp64" if kind == "grad" else rng.choice(("df32", "df32", "fp64", "fp64", "fp32"))
        if kind != "sweep" and prec == "fp32":
            continue
        n_groups = rng.choice((1, 1, 1, 2, 3)) if kind == "sweep" else 1
        gs = []
        for _ in range(n_groups):
            Lx = 2 * rng.randint(1, 8)
            Ly = rng.choice((Lx, Lx, 2 * rng.randint(1, 8)))
            dtau = rng.choice((0.4, 0.25, 0.2, 0.125, 0.1))
            L = rng.randint(10, 160)
            chains = int(round(2 ** rng.uniform(0, 9)))
            span = 0.25 if prec == "fp32" else rng.uniform(0.8, 1.3)
            ns = max(1, int(round(span / dtau)))
            gs.append(_g(Lx, Ly, rng.choice((0.5, 1.0, 2.0, 3.0)), L * dtau, dtau, chains, ns,
                         rng.choice((8, 16, 16, 32, rng.randint(4, 32)))))
        case = dict(kind=kind, precision=prec, groups="; ".join(gs))
        if kind == "sweep":
            case["gtau"] = rng.random() < 0.5
        if kind == "origins":
            case["origins"] = rng.randint(2, 4)
        groups = _groups(case)
        cost = _cost(groups, case.get("gtau")) * case.get("origins", 1)
        decisions = sum(g.N * g.L * g.n_chains for g in groups)
        # FP32 decisions follow its rounding error: few of them, so that the chains stay the same
        if cost < 0.3 and not (prec == "fp32" and decisions > 200_000):
            return case


def _groups(case):
    out = []
    for text in case["groups"].split(";"):
        size, U, beta, dtau, chains, ns, k = text.split(",")
        Lx, Ly = size.split("x")
        out.append(pkg.Group(Lx=int(Lx), Ly=int(Ly), t=T_HOP, U=float(U), beta=float(beta),
                             dtau=float(dtau), n_chains=int(chains), stab_interval=int(ns),
                             delay_k=int(k), precision=case["precision"]))
    return out


# ---------------------------------------------------------------------------
# What a program holds before the call, and the call.
# ---------------------------------------------------------------------------
def _runs(case, seed):
    """G_k(tau)-like runs: a decay per momentum with a dtau^2 error and chain noise."""
    N, beta = case["Lx"] * case["Ly"], case["beta"]
    slices = [int(s) for s in case["slices"].split(",")]
    rng = np.random.default_rng(seed)
    eps = rng.uniform(-1.0, 1.0, N)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    runs = []
    for L in slices:
        tau = np.arange(L + 1) * (beta / L)
        g = np.exp(-np.outer(tau, eps)) / (1.0 + np.exp(-beta * eps)) * (1.0 + 0.3 * (beta / L) ** 2)
        noise = torch.randn((case["chains"], L + 1, N), dtype=torch.float64, device="cuda", generator=gen)
        runs.append(torch.from_numpy(g).cuda() + 0.05 * noise)
    return [beta / L for L in slices], runs


def _fields(groups, seed):
    rng = np.random.default_rng(seed)
    return [(2 * rng.integers(0, 2, (g.n_chains, g.L, g.N)) - 1).astype(np.int8) for g in groups]


def prepare(case, seed):
    if case["kind"] == "analysis":
        dtaus, runs = _runs(case, seed)
        return dict(case=case, dtaus=dtaus, runs=runs)
    groups = _groups(case)
    s = dict(case=case, groups=groups, sim=pkg.DQMC(groups, seed=seed))
    n = sum(g.n_chains * (g.L + 1) * g.N for g in groups)
    if case.get("gtau") or case["kind"] == "origins":
        s["buf"] = torch.empty(n, dtype=torch.float64, device="cuda")
    if case["kind"] == "green":
        s["fields"] = _fields(groups, seed)
    if case["kind"] == "grad":
        g = groups[0]
        s["t"] = torch.tensor(g.t, dtype=torch.float64, requires_grad=True)
        s["lam"] = torch.tensor(math.acosh(math.exp(0.5 * g.dtau * g.U)), dtype=torch.float64,
                                requires_grad=True)
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "analysis":
        fine = pkg.trotter_extrapolate(s["dtaus"], s["runs"], case["beta"], case["fine"])
        g_iw, sigma = pkg.matsubara_sigma(fine, case["beta"], case["Lx"], case["Ly"], T_HOP, case["freqs"])
        return dict(fine=fine, g_iw=g_iw, sigma=sigma)
    sim = s["sim"]
    out = {}
    if case["kind"] == "green":
        sim.set_field(s["fields"])
        out["G"] = np.stack([[sim.G(c, spin) for spin in (0, 1)] for c in range(sim.n_chains)])
        return out
    if case["kind"] == "origins":
        out["gtau"] = sim.gtau_origins(case["origins"], out=s["buf"])
        return out
    sim.sweep(1, measure=True)
    if case["kind"] == "grad":
        s["t"].grad = s["lam"].grad = None
        lw = pkg.LogWeight.apply(sim, s["t"], s["lam"])
        lw.sum().backward()
        out["logw"], out["dt"], out["dlam"] = lw.detach(), s["t"].grad, s["lam"].grad
    elif case["gtau"]:
        out["gtau"] = sim.gtau(out=s["buf"])
    out["field"] = sim.field()
    out["observables"] = sim.observables()
    out["spin"] = sim.spin_correlation()
    out["accepted"] = sim.stats()[1].astype(np.int64)
    if sim.n_chains <= 8:
        out["G"] = np.stack([sim.G(c) for c in range(sim.n_chains)])
    return out


# ---------------------------------------------------------------------------
# What a step cannot do without.
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "analysis":
        N, M, F = case["Lx"] * case["Ly"], case["fine"], case["freqs"]
        rows = sum(int(x) + 1 for x in case["slices"].split(","))
        R = len(case["slices"].split(","))
        return dict(bytes=8 * N * (case["chains"] * rows + (M + 1) + 4 * F),
                    flops=N * (case["chains"] * rows + 12 * rows + 12 * R * M + 8.0 * F * M))
    flops = nbytes = 0.0
    for g in _groups(case):
        N, L, C, nc = g.N, g.L, g.n_chains, math.ceil(g.L / g.stab_interval)
        kron = 2.0 * L * N * N * (g.Lx + g.Ly)  # one pass of B_L ... B_1 over N vectors
        # a pass over one UDT stack: Kronecker products, QR with Q, triangular update of T
        stack = kron + nc * (8.0 / 3 + 1.0) * N ** 3
        point = (2 * 2 + 2) * N ** 3  # two products for the middle matrix, its inverse
        wrap = 2 * kron
        f = 0.0
        if case["kind"] in ("sweep", "grad"):
            # half of the proposals accepted, one rank-1 update of G each
            f += L * N * 0.5 * 2.0 * N * N + wrap + 2 * stack + nc * (point + 4.0 * N ** 3)
        if case["kind"] == "grad":
            f += (nc + 1) * (point + 4.0 * N ** 3) + wrap
        if case.get("gtau"):
            f += (nc + 1) * (point + 8.0 * N ** 3) + 2 * kron
        if case["kind"] == "green":
            f += 2 * stack + point + 4.0 * N ** 3
        if case["kind"] == "origins":
            n = case["origins"]
            f += n * (2 * stack + (nc + 1) * (point + 8.0 * N ** 3) + 2 * kron)
        flops += C * f
        # the field, the working G and the two stacks (U, T) read or written once
        nbytes += C * (2 * L * N + 2 * 8 * N * N + 4 * 8 * (nc + 1) * N * N)
        if case.get("gtau") or case["kind"] == "origins":
            nbytes += 8 * C * (L + 1) * N
    return dict(bytes=nbytes, flops=flops)


# ---------------------------------------------------------------------------
# The same results in plain numpy FP64 (Rost & Bluemer, arXiv:1504.05090,
# Eqs. (1)-(3)); Philox4x32-10 after Salmon et al., SC'11.
# ---------------------------------------------------------------------------
_SUB = 4  # slices between two orthogonalisations


def _philox(c, seed):
    c = [np.asarray(x, dtype=np.uint64) for x in np.broadcast_arrays(*c)]
    m32 = np.uint64(0xFFFFFFFF)
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64((seed >> 32) & 0xFFFFFFFF)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & m32]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
    return c


def _T(x):
    return np.swapaxes(x, -1, -2)


class _Model:
    """One group of chains, all of them at once: arrays [chain, ...]."""

    def __init__(self, g, chain0, seed, field=None):
        self.g, self.seed, self.N, self.L, self.C = g, seed, g.N, g.L, g.n_chains
        self.chains = chain0 + np.arange(self.C)
        N, Lx, Ly = self.N, g.Lx, g.Ly
        i = np.arange(N)
        x, y = i % Lx, i // Lx
        self.A = np.zeros((N, N))
        for nb in ((x + 1) % Lx + Lx * y, (x - 1) % Lx + Lx * y, x + Lx * ((y + 1) % Ly),
                   x + Lx * ((y - 1) % Ly)):
            np.add.at(self.A, (i, nb), 1.0)
        w, v = np.linalg.eigh(self.A)
        self.E = (v * np.exp(g.dtau * T_HOP * w)) @ v.T
        self.Ei = (v * np.exp(-g.dtau * T_HOP * w)) @ v.T
        self.lam = math.acosh(math.exp(0.5 * g.dtau * g.U))
        self.P = np.where((x + y) % 2 == 0, 1.0, -1.0)
        # to[r, i]: the site i + r
        self.to = (x[None] + x[:, None]) % Lx + Lx * ((y[None] + y[:, None]) % Ly)
        self.cp = sorted(set(range(0, self.L, g.stab_interval)) | {self.L})
        self.pts = sorted({p for a, b in zip(self.cp, self.cp[1:]) for p in range(a, b, _SUB)} | {self.L})
        if field is None:
            e = np.arange(self.L * N)
            r = _philox((e[None], 0xFFFFFFFF, self.chains[:, None], 1), seed)[0]
            field = np.where(r & np.uint64(1), 1, -1).reshape(self.C, self.L, N)
        self.s = field.astype(np.float64)

    def ev(self, l, sg):
        return np.exp(sg * self.lam * self.s[:, l])

    def _udt(self, X, T):
        order = np.argsort(-np.sum(X * X, axis=1), axis=1)
        Q, R = np.linalg.qr(np.take_along_axis(X, order[:, None], axis=2))
        D = np.abs(np.diagonal(R, axis1=1, axis2=2)).copy()
        back = np.argsort(order, axis=1)
        return Q, D, np.take_along_axis(R / D[:, :, None], back[:, None], axis=2) @ T

    def _one(self):
        return (np.broadcast_to(np.eye(self.N), (self.C, self.N, self.N)), np.ones((self.C, self.N)),
                np.broadcast_to(np.eye(self.N), (self.C, self.N, self.N)))

    def right(self, a, b, udt, sg):
        X = udt[0] * udt[1][:, None]
        for l in range(a, b):
            X = self.E @ (self.ev(l, sg)[:, :, None] * X)
        return self._udt(X, udt[2])

    def lefts(self, sg):
        out = {self.L: self._one()}
        for a, b in zip(self.pts[-2::-1], self.pts[:0:-1]):
            u, d, t = out[b]
            X = u * d[:, None]
            for l in range(b - 1, a - 1, -1):
                X = self.ev(l, sg)[:, :, None] * (self.E @ X)
            out[a] = self._udt(X, t)
        return out

    def solve(self, R, Lf):
        """U_L Db_L^-1 Mid^-1 and G of one point."""
        (ur, dr, tr), (ul, dl, tl) = R, Lf
        br, bl, sr, sl = np.maximum(dr, 1), np.maximum(dl, 1), np.minimum(dr, 1), np.minimum(dl, 1)
        mid = (_T(ur) @ ul) / br[:, :, None] / bl[:, None] + sr[:, :, None] * (tr @ _T(tl)) * sl[:, None]
        W = (ul / bl[:, None]) @ np.linalg.inv(mid)
        return W, (W / br[:, None]) @ _T(ur), mid

    def wrap(self, G, l, sg=1):
        e = self.ev(l, sg)
        return self.E @ (e[:, :, None] * G / e[:, None]) @ self.Ei

    def down(self, G):
        return np.eye(self.N) - self.P[:, None] * _T(G) * self.P

    def sweep(self, number):
        N, g = self.N, self.g
        em, ep = math.expm1(-2 * self.lam), math.expm1(2 * self.lam)
        Lf, R, j = self.lefts(1), self._one(), 0
        G = self.solve(R, Lf[0])[1].copy()
        obs, spin = np.zeros((self.C, 4)), np.zeros((self.C, N))
        ar = np.arange(N)
        for l in range(self.L):
            w = _philox((ar[None] + N * l, number, self.chains[:, None], 0), self.seed)
            u = ((w[0] << np.uint64(32) | w[1]) >> np.uint64(11)).astype(np.float64) * 2.0 ** -53
            for i in range(N):
                gi, s = G[:, i, i], self.s[:, l, i]
                du, dd = np.where(s > 0, em, ep), np.where(s > 0, ep, em)
                ru = 1 + du * (1 - gi)
                ok = np.nonzero(u[:, i] < ru * (1 + dd * gi))[0]
                if len(ok):
                    H = G[ok]
                    col = -H[:, :, i]
                    col[:, i] += 1
                    G[ok] = H - (du[ok] / ru[ok])[:, None, None] * col[:, :, None] * H[:, i][:, None]
                    self.s[ok, l, i] *= -1
            G = self.wrap(G, l)
            if l + 1 in Lf:
                R = self.right(self.pts[j], l + 1, R, 1)
                G = self.solve(R, Lf[l + 1])[1].copy()
                j += 1
                if l + 1 in self.cp:
                    self._measure(G, obs, spin)
        return obs, spin, G

    def _measure(self, G, obs, spin):
        N, eye = self.N, np.eye(self.N)
        Gd = self.down(G)
        nu, nd = 1 - np.diagonal(G, axis1=1, axis2=2), 1 - np.diagonal(Gd, axis1=1, axis2=2)
        obs[:, 0] += (nu + nd).mean(1)
        obs[:, 1] += (nu * nd).mean(1)
        obs[:, 2] += -T_HOP * sum(np.sum(self.A * (eye - _T(x)), axis=(1, 2)) for x in (G, Gd)) / N
        obs[:, 3] += 1
        m = nu - nd
        ss = m[:, :, None] * m[:, None] + sum((eye - _T(x)) * x for x in (G, Gd))
        spin += np.stack([ss[:, np.arange(N), self.to[r]].mean(1) for r in range(N)], axis=1) / 4

    def gtau(self):
        N, g, out = self.N, self.g, 0.0
        ar = np.arange(N)
        for sg in (1, -1):
            Lf, R, rows = self.lefts(sg), self._one(), []
            for q, p in enumerate(self.pts):
                X = self.solve(R, Lf[p])[0] * np.minimum(R[1], 1)[:, None] @ R[2]
                end = self.pts[q + 1] if q + 1 < len(self.pts) else self.L + 1
                for l in range(p, end):
                    if l > p:
                        X = self.E @ (self.ev(l - 1, sg)[:, :, None] * X)
                    r = np.stack([X[:, self.to[d], ar].mean(1) for d in range(N)], axis=1)
                    rows.append(np.fft.fft2(r.reshape(-1, g.Ly, g.Lx)).real.reshape(-1, N))
                if q + 1 < len(self.pts):
                    R = self.right(p, self.pts[q + 1], R, sg)
            out = out + 0.5 * np.stack(rows, axis=1)
        return out

    def grad(self):
        Lf, R, dt, dl = self.lefts(1), self._one(), 0.0, 0.0
        eye = np.eye(self.N)
        for q, p in enumerate(self.pts):
            _, G, mid = self.solve(R, Lf[p])
            if q == 0:
                lw = np.linalg.slogdet(mid)[1] + np.sum(np.log(np.maximum(Lf[0][1], 1)), axis=1)
                lw = 2 * lw - self.lam * self.s.sum((1, 2))
            end = self.pts[q + 1] if q + 1 < len(self.pts) else p
            for l in range(p, end):  # G(l); slice l + 1 follows
                dl = dl + np.sum(self.s[:, l] * (1 - 2 * np.diagonal(G, axis1=1, axis2=2)), axis=1)
                dt = dt + self.g.dtau * sum(np.sum(self.A * (eye - _T(x)), axis=(1, 2))
                                            for x in (G, self.down(G)))
                G = self.wrap(G, l)
            if q + 1 < len(self.pts):
                R = self.right(p, self.pts[q + 1], R, 1)
        # the sum over l = 1 .. L equals that over l = 0 .. L - 1: G(L) = G(0)
        return dt, dl, lw


def _spline_moments(y, h):
    """Second derivatives of the not-a-knot cubic spline through y[m] on a uniform grid."""
    n = len(y) - 1
    M = np.zeros((n + 1, n + 1))
    rhs = np.zeros_like(y)
    for m in range(1, n):
        M[m, m - 1:m + 2] = 1.0, 4.0, 1.0
    rhs[1:n] = 6.0 / h ** 2 * (y[2:] - 2 * y[1:-1] + y[:-2])
    M[0, :3] = M[n, n - 2:] = 1.0, -2.0, 1.0
    return np.linalg.solve(M, rhs)


def _spline(y, h, x):
    z = _spline_moments(y, h)
    m = np.clip((x / h).astype(int), 0, len(y) - 2)
    b = (x / h - m)[:, None]
    a = 1 - b
    return a * y[m] + b * y[m + 1] + ((a ** 3 - a) * z[m] + (b ** 3 - b) * z[m + 1]) * h ** 2 / 6


def _exact_analysis(case, seed):
    beta, M, Lx, Ly = case["beta"], case["fine"], case["Lx"], case["Ly"]
    dtaus, runs = _runs(case, seed)
    tau = np.arange(M + 1) * (beta / M)
    ys = np.stack([_spline(r.mean(0).cpu().numpy(), dt, tau) for dt, r in zip(dtaus, runs)])
    x = np.array(dtaus) ** 2
    if len(x) == 1:
        fine = ys[0]
    else:
        xc = x - x.mean()
        slope = np.tensordot(xc, ys, 1) / np.sum(xc * xc)
        fine = ys.mean(0) - slope * x.mean()
    nodes, wts = np.polynomial.legendre.leggauss(14)
    h = beta / M
    t = (np.arange(M)[:, None] + 0.5 * (nodes + 1)[None]).ravel() * h
    wt = np.tile(0.5 * h * wts, M)
    om = (2 * np.arange(case["freqs"]) + 1) * math.pi / beta
    g_iw = -(np.exp(1j * np.outer(om, t)) * wt) @ _spline(fine, h, t)
    kx, ky = np.arange(Lx * Ly) % Lx, np.arange(Lx * Ly) // Lx
    eps = -2 * T_HOP * (np.cos(2 * np.pi * kx / Lx) + np.cos(2 * np.pi * ky / Ly))
    return dict(fine=fine, g_iw=g_iw, sigma=1j * om[:, None] - eps - 1 / g_iw)


def exact(case, seed):
    if case["kind"] == "analysis":
        return _exact_analysis(case, seed)
    groups = _groups(case)
    spins = 2 if case.get("gtau") or case["kind"] == "origins" else 1
    cost = 0.0
    for g in groups:
        cost += g.n_chains * g.L * (g.N ** 3 * 2.5e-9 * spins + g.N * 6e-6) * case.get("origins", 1)
        if case["kind"] in ("sweep", "grad"):
            cost += g.L * g.N * (5e-5 + g.n_chains * g.N ** 2 * 3e-9)
    if cost > 15.0:
        return None
    fields = _fields(groups, seed) if case["kind"] == "green" else [None] * len(groups)
    out, chain = {}, 0
    parts = []
    for g, f in zip(groups, fields):
        parts.append(_Model(g, chain, seed, f))
        chain += g.n_chains
    if case["kind"] == "green":
        G = [m.solve(m._one(), m.lefts(1)[0])[1] for m in parts]
        return dict(G=np.concatenate([np.stack([x, m.down(x)], axis=1) for m, x in zip(parts, G)]))
    if case["kind"] == "origins":
        flat = []
        for m in parts:
            s0, acc = m.s, 0.0
            for o in range(case["origins"]):
                m.s = np.roll(s0, -((o * m.L) // case["origins"]), axis=1)
                acc = acc + m.gtau() / case["origins"]
            flat.append(acc.ravel())
        return dict(gtau=np.concatenate(flat))
    done = [m.sweep(0) for m in parts]
    if case["kind"] == "grad":
        dt, dl, lw = (np.concatenate(v) for v in zip(*(m.grad() for m in parts)))
        out.update(logw=lw, dt=np.float64(dt.sum()), dlam=np.float64(dl.sum()))
    elif case["gtau"]:
        out["gtau"] = np.concatenate([m.gtau().ravel() for m in parts])
    out["field"] = [None] * len(parts)
    out["observables"] = np.concatenate([d[0] for d in done])
    out["spin"] = [d[1] for d in done]
    out["accepted"] = None
    if chain <= 8:
        out["G"] = np.stack([x for d in done for x in d[2]])
    return out
