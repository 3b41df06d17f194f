"""Performance cases of the library: what a simulation run asks of it, from the first field to the last.

A pass of every case is a run as a program makes it through the public binding: ``init_fields`` from
page-locked host arrays, a number of time steps, ``read_fields`` into page-locked host arrays (with
the film statistics or the conservation checks in between where that kind of run has them). Contexts
and batches are created once and used for many runs; the fields of a run come from its seed.

``exact`` is the same run in plain 64-bit torch: the method's equations on whole arrays.
"""
import math

import numpy as np
import torch

from paper_2603_17481_gb300 import binding as B
from paper_2603_17481_gb300 import workloads as W

STORE_BYTES = {"f32": 4, "f16": 2, "bf16": 2}


# --------------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------------

def listed():
    return [
        # The 2D head-on collision of the paper's planar set-up, the smallest run: a few microseconds of
        # work per kernel, so launches and latency count.
        dict(name="drops_2d_128x64", kind="drops", dim=2, nx=128, ny=64, nz=1, Q=9, store="f32", R=16.0,
             ratio=1.0, steps=200),
        # A 2D run of production size on a grid no tile divides.
        dict(name="drops_2d_1021x509", kind="drops", dim=2, nx=1021, ny=509, nz=1, Q=9, store="f32", R=96.0,
             ratio=10.0, steps=200),
        # A small 3D run that is watched: the conservation check runs every ten steps.
        dict(name="watched_48x48x48", kind="drops", dim=3, nx=48, ny=48, nz=48, Q=19, store="f32", R=8.0,
             ratio=10.0, steps=200, check=10),
        # The off-centre collision used for validation; its state fits the L2 cache.
        dict(name="drops_128x64x64", kind="drops", dim=3, nx=128, ny=64, nz=64, Q=19, store="f32", R=12.0,
             ratio=10.0, steps=200),
        # An odd, ragged 3D box: rows of odd length and partial tiles on every side.
        dict(name="drops_107x75x61", kind="drops", dim=3, nx=107, ny=75, nz=61, Q=19, store="f32", R=13.0,
             ratio=10.0, steps=200),
        # The benchmark collision at density ratio 100, plain FP32 populations.
        dict(name="drops_256x128x128", kind="drops", dim=3, nx=256, ny=128, nz=128, Q=19, store="f32", R=24.0,
             ratio=100.0, steps=200),
        # The same with FP16 populations, the storage for runs that want throughput.
        dict(name="drops_256x128x128_f16", kind="drops", dim=3, nx=256, ny=128, nz=128, Q=19, store="f16",
             R=24.0, ratio=100.0, steps=200),
        # The paper's own lattice, D3Q27.
        dict(name="drops_160x96x96_q27", kind="drops", dim=3, nx=160, ny=96, nz=96, Q=27, store="f32", R=18.0,
             ratio=100.0, steps=100),
        # The parameter sweep: uneven collisions advanced together as one batch.
        dict(name="sweep_24", kind="sweep", cases=24, store="f32", steps=50),
        # The film sweep: a batch of head-on collisions close to contact whose film statistics are taken
        # every 20 steps.
        dict(name="films_9", kind="films", cases=9, store="f32", steps=60),
        # The buoyant bubble swarm at the bubble density of the 512^3 one, the largest run: interfaces in a
        # third of the tiles.
        dict(name="swarm_384", kind="swarm", L=384, Q=19, store="f32", steps=40),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["2d", "3d", "3d", "3d", "3d", "sweep", "films", "swarm"])
    store = rng.choice(["f32", "f32", "f16", "bf16"])
    if kind == "2d":
        nx, ny = int(_log(rng, 64, 1200)), int(_log(rng, 48, 640))
        return dict(kind="drops", dim=2, nx=nx, ny=ny, nz=1, Q=9, store=store, R=round(min(nx, 2 * ny) / 8.0, 2),
                    ratio=rng.choice([1.0, 10.0, 100.0]), steps=rng.randrange(60, 241))
    if kind == "sweep":
        return dict(kind="sweep", cases=rng.randrange(8, 33), store=store, steps=rng.randrange(20, 61))
    if kind == "films":
        return dict(kind="films", cases=rng.randrange(4, 13), store=store, steps=20 * rng.randrange(2, 5))
    if kind == "swarm":
        return dict(kind="swarm", L=4 * rng.randrange(24, 81), Q=19, store=store, steps=rng.randrange(20, 41))
    side = _log(rng, 44, 160)  # cells: 44^3 to 160^3
    ax, ay = rng.uniform(1.0, 2.0), rng.uniform(0.8, 1.25)
    n = [max(32, int(v)) for v in (side * ax / ax ** (1 / 3), side * ay / (ax ** (1 / 3) * ay ** 0.5),
                                   side / (ax ** (1 / 3) * ay ** 0.5))]
    if rng.random() < 0.6:  # the grids people choose: rows of a multiple of 8
        n = [8 * max(4, round(v / 8)) for v in n]
    return dict(kind="drops", dim=3, nx=n[0], ny=n[1], nz=n[2], Q=rng.choice([19, 19, 19, 27]), store=store,
                R=round(min(n[0] / 8.0, min(n[1:]) / 4.0), 2), ratio=rng.choice([10.0, 100.0]),
                steps=rng.randrange(60, 201), check=rng.choice([0, 0, 0, 10]))


# --------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------

def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _drops_cfg(case, rng):
    """Two droplets on a collision course (one above the other axis by a seeded offset)."""
    dim, nx, ny, nz, R = case["dim"], case["nx"], case["ny"], case["nz"], case["R"]
    cfg = W.base_config(dim, nx, ny, nz, case["Q"], rho_g=1.0 / case["ratio"])
    gap, off, speed = rng.uniform(6.0, 10.0), rng.uniform(0.0, 0.5) * R, rng.uniform(0.03, 0.05)
    c = [(nx - 1) / 2.0, (ny - 1) / 2.0, (nz - 1) / 2.0]
    sep = 2 * R + gap
    cfg.update(R=R, centers=[(c[0] - sep / 2, c[1] - off / 2, c[2]), (c[0] + sep / 2, c[1] + off / 2, c[2])],
               velocities=[(speed / 2, 0.0, 0.0), (-speed / 2, 0.0, 0.0)])
    return cfg


def _films_cfgs(n, rng):
    """Head-on collisions over D x sigma x A_rep / sigma whose films are about to form."""
    grid = [(D, sg, r) for r in (1.0, 0.5, 2.0) for sg in (0.01, 0.005, 0.02) for D in (24, 32, 48)]
    out = []
    for D, sg, r in grid[:n]:
        cfg = W.selftune_cases((D,), (sg,), (r,))[0]
        gap = rng.uniform(2.5, 5.0)
        (a, y, z), (b, _, _) = cfg["centers"]
        mid, sep, (dy, dz) = 0.5 * (a + b), 2 * cfg["R"] + gap, rng.uniform(-0.5, 0.5, 2)
        cfg["centers"] = [(mid - sep / 2, y, z), (mid + sep / 2, y + dy, z + dz)]
        out.append(cfg)
    return out


def _configs(case, seed):
    """The configurations of a case's simulations (one, or one per batched case)."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "drops":
        return [_drops_cfg(case, rng)]
    if case["kind"] == "sweep":
        # the sweep's grids, each with a Weber number and an impact offset of this seed
        return [W.collision_sweep(1, seed=int(rng.integers(1 << 30)), grids=(c["nx"],))[0]
                for c in W.collision_sweep(case["cases"])]
    if case["kind"] == "films":
        return _films_cfgs(case["cases"], rng)
    L = case["L"]
    cfg = W.base_config(3, L, L, L, case["Q"], rho_g=0.01, sigma=0.01, nu_l=1e-3, nu_g=1e-2, A_rep=0.01,
                        g=(0.0, 0.0, -1e-6))
    # bubbles of radius 8 to 12, at least two interface widths apart, at the density of 1500 in 512^3
    nb, cs, rs = max(2, round(1500 * (L / 512.0) ** 3)), np.zeros((0, 3)), np.zeros(0)
    while len(rs) < nb:
        c, r = rng.uniform(0.0, L, 3), rng.uniform(8.0, 12.0)
        d = cs - c
        d -= L * np.round(d / L)
        if np.all((d * d).sum(1) >= (rs + r + 2 * cfg["eps"]) ** 2):
            cs, rs = np.vstack([cs, c]), np.append(rs, r)
    cfg.update(centers=cs.tolist(), radii=rs.tolist())
    return [cfg]


def _fields(cfg, dev):
    """phi (on the fixed-point grid) and u (3, N) in FP64: tanh droplets, or tanh bubbles at rest."""
    n = (cfg["nx"], cfg["ny"], cfg["nz"])
    N = n[0] * n[1] * n[2]
    ax = [torch.arange(k, dtype=torch.float64, device=dev) for k in n]

    def dist(c, idx):
        d = []
        for a in range(3):
            x = ax[a][idx[a]] - c[a] if idx else ax[a] - c[a]
            d.append(x - n[a] * torch.round(x / n[a]) if a < cfg["dim"] else 0.0 * x)
        return torch.sqrt(d[2][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[0][None, None, :] ** 2)

    u = torch.zeros(3, N, dtype=torch.float64, device=dev)
    acc = torch.zeros(n[2], n[1], n[0], dtype=torch.float64, device=dev)
    if "radii" in cfg:  # bubble by bubble, within 4 interface widths of its surface
        for c, R in zip(cfg["centers"], cfg["radii"]):
            h = int(math.ceil(R + 4 * cfg["eps"]))
            idx = [(torch.arange(2 * h + 2, device=dev) + int(c[a]) - h) % n[a] for a in range(3)]
            r = dist(c, idx)
            prof = 0.5 * (1.0 + torch.tanh(2.0 * (R - r) / cfg["eps"]))
            prof[r > R + 4 * cfg["eps"]] = 0.0
            acc[idx[2][:, None, None], idx[1][None, :, None], idx[0][None, None, :]] += prof
        phi = torch.clamp(1.0 - acc, min=0.0)
    else:
        for c, U in zip(cfg["centers"], cfg["velocities"]):
            prof = 0.5 * (1.0 + torch.tanh(2.0 * (cfg["R"] - dist(c, None)) / cfg["eps"]))
            acc += prof
            for a in range(cfg["dim"]):
                u[a] += prof.reshape(-1) * U[a]
        phi = torch.clamp(acc, max=1.0)
    return torch.round(phi.reshape(-1) * W.Q30) / W.Q30, u


def _host(*shape):
    return torch.zeros(*shape, dtype=torch.float64, pin_memory=torch.cuda.is_available())


def prepare(case, seed):
    cfgs = _configs(case, seed)
    sizes = [W.ncells(c) for c in cfgs]
    at = np.concatenate([[0], np.cumsum(sizes)])
    total = int(at[-1])
    # one page-locked block per field, a slice per simulation
    blocks = [_host(total), _host(3 * total), _host(total), _host(3 * total), _host(total)]
    views = []
    for k in range(len(cfgs)):
        lo, hi = int(at[k]), int(at[k + 1])
        views.append([b[w * lo:w * hi] for b, w in zip(blocks, (1, 3, 1, 3, 1))])
    for cfg, v in zip(cfgs, views):
        phi, u = _fields(cfg, _dev())
        v[0].copy_(phi)
        v[1].copy_(u.reshape(-1))
    sims = [B.Lbm(c, store=case["store"], mass_check_every=case.get("check", 0)) for c in cfgs]
    state = dict(case=case, sims=sims, views=views, out=blocks[2:], batch=None)
    if len(sims) > 1:  # a batch takes initialised contexts
        for s, v in zip(sims, views):
            s.init_fields(v[0], v[1])
        state["batch"] = B.LbmBatch(sims, nstreams=16)
    return state


def run(state):
    case, sims, views, batch = state["case"], state["sims"], state["views"], state["batch"]
    steps = case["steps"]
    films = []
    for s, v in zip(sims, views):
        s.init_fields(v[0], v[1])
    if batch is None:
        sims[0].step(steps)
    elif case["kind"] == "films":
        for _ in range(0, steps, 20):
            batch.step(20)
            films.append([list(s.nci_diagnostics().values()) for s in sims])
    else:
        batch.step(steps)
    for s, v in zip(sims, views):
        s.read_fields(phi=v[2], u=v[3], pstar=v[4])
    phi, u, ps = state["out"]
    return dict(phi=phi, u=u, pstar=ps, **({"films": np.array(films)} if films else {}))


def work(case):
    """One pass: the fields in (phi, u) and out (phi, u, p*) as FP64, and per step each population and
    phi read once and written once; operations of the collision and of the phase-field update."""
    cells = [W.ncells(c) for c in _configs(case, 1)] if case["kind"] in ("sweep", "films") else (
        [case["L"] ** 3] if case["kind"] == "swarm" else [case["nx"] * case["ny"] * case["nz"]])
    N, Q = sum(cells), case.get("Q", 19)
    return {"bytes": N * (72.0 + case["steps"] * (2.0 * Q * STORE_BYTES[case["store"]] + 8.0)),
            "flops": N * case["steps"] * (30.0 * Q + 250.0)}


# --------------------------------------------------------------------------------------------
# The same run in 64 bits
# --------------------------------------------------------------------------------------------

class _Exact:
    """The method on whole FP64 arrays of shape (nz, ny, nx) (leading axis: component or direction)."""

    def __init__(self, cfg, dev):
        self.p, self.dev, self.dim = cfg, dev, cfg["dim"]
        self.shape = (cfg["nz"], cfg["ny"], cfg["nx"])
        wt = {9: {0: 4 / 9, 1: 1 / 9, 2: 1 / 36}, 19: {0: 1 / 3, 1: 1 / 18, 2: 1 / 36},
              27: {0: 8 / 27, 1: 2 / 27, 2: 1 / 54, 3: 1 / 216}}[cfg["Q"]]
        z = (0,) if self.dim == 2 else (-1, 0, 1)
        c = [(a, b, d) for d in z for b in (-1, 0, 1) for a in (-1, 0, 1) if a * a + b * b + d * d in wt]
        self.c = c
        self.w = [wt[a * a + b * b + d * d] for a, b, d in c]

    def at(self, f, a, k):  # f at x + k e_a
        return torch.roll(f, -k, 2 - a) if a < self.dim else f

    def smooth(self, f, but=-1):
        for a in range(self.dim):
            if a != but:
                f = (self.at(f, a, 1) + self.at(f, a, -1) + 4.0 * f) / 6.0
        return f

    def d(self, f, a):  # isotropic derivative along a
        return 0.5 * self.smooth(self.at(f, a, 1) - self.at(f, a, -1), a)

    def grad(self, f):
        return [self.d(f, a) if a < self.dim else torch.zeros_like(f) for a in range(3)]

    def normal(self, g):
        s = torch.sqrt(g[0] ** 2 + g[1] ** 2 + g[2] ** 2) + self.p["eps_n"]
        return [x / s for x in g]

    def repulsion(self, phi, g):
        """F_rep (3 arrays) and the cells that have a partner (flat indices)."""
        p, (nz, ny, nx) = self.p, self.shape
        F = torch.zeros((3,) + self.shape, dtype=torch.float64, device=self.dev)
        pc = phi.clamp(0.0, 1.0)
        q = (pc * (1.0 - pc)).reshape(-1)
        cells = torch.nonzero(q >= p["q_th"]).reshape(-1)
        n = torch.stack([x.reshape(-1) for x in self.normal(g)])
        w, zr = p["w"], p["w"] if self.dim == 3 else 0
        r = torch.tensor([(a, b, d) for d in range(-zr, zr + 1) for b in range(-w, w + 1) for a in range(-w, w + 1)
                          if (a, b, d) != (0, 0, 0)], device=self.dev)
        d2 = (r * r).sum(1)
        order = torch.argsort(d2, stable=True)  # by distance, then by window index
        r, d2 = r[order], d2[order].double()
        hit = []
        for part in torch.split(cells, 1 << 18):
            x, y, z = part % nx, (part // nx) % ny, part // (nx * ny)
            m = ((x[:, None] + r[:, 0]) % nx) + nx * (((y[:, None] + r[:, 1]) % ny)
                                                      + ny * ((z[:, None] + r[:, 2]) % nz))
            dot = n[0][part][:, None] * n[0][m]
            dot += n[1][part][:, None] * n[1][m]
            dot += n[2][part][:, None] * n[2][m]
            qm, qx = q[m], q[part][:, None]
            ok = (qm >= p["q_th"]) & ((qm - qx).abs() <= p["eta"] * qx.clamp(min=p["eps_q"])) & (dot <= p["cos_opp"])
            # nearest first, then the largest facing score, then the first in the window
            key = torch.where(ok, d2 * 4.0 + dot, torch.inf)
            best = torch.argmin(key, 1)
            have = torch.nonzero(torch.isfinite(key.gather(1, best[:, None])[:, 0])).reshape(-1)
            if len(have):
                hit.append((part[have], m[have, best[have]], r[best[have]].double().T, -dot[have, best[have]]))
        if not hit:
            return F, cells[:0]
        i, j = (torch.cat([h[k] for h in hit]) for k in (0, 1))
        off, ff = torch.cat([h[2] for h in hit], 1), torch.cat([h[3] for h in hit])
        qcl = (0.5 * (q[i] + q[j])).clamp(p["eps_q"], 0.25 - p["eps_q"])
        h = p["eps"] * torch.acosh(1.0 / (2.0 * torch.sqrt(qcl)))
        wh = 1.0 / (1.0 + (h / p["h0"]) ** p["p"])
        s = n[:, i] - n[:, j]
        s = s / (s.norm(dim=0) + p["eps_n"])
        s = torch.where((s * off).sum(0) < 0.0, -s, s)
        amp = (p["rho_g"] + (p["rho_l"] - p["rho_g"]) * phi.reshape(-1)[i]) * p["A_rep"] * qcl * wh * ff
        for a in range(self.dim):
            F[a].view(-1)[i] = amp * s[a]
        return F, i

    def chemical(self, phi):
        p = self.p
        beta, kap = 12.0 * p["sigma"] / p["eps"], 1.5 * p["sigma"] * p["eps"]
        return 4.0 * beta * phi * (phi - 1.0) * (phi - 0.5) - kap * 6.0 * (self.smooth(phi) - phi)

    def hydro(self, f, phi, post):
        """u and p* of the pre-collision populations; with post, f becomes the streamed f_post."""
        p, dim = self.p, range(self.dim)
        dr = p["rho_l"] - p["rho_g"]
        rho = p["rho_g"] + dr * phi
        g = self.grad(phi)
        nu = (p["rho_g"] * p["nu_g"] + (p["rho_l"] * p["nu_l"] - p["rho_g"] * p["nu_g"]) * phi) / rho
        om = 1.0 / (0.5 + 3.0 * nu)
        mu = self.chemical(phi)
        rep = self.repulsion(phi, g)[0] if p["nci_on"] else torch.zeros((3,) + self.shape, device=self.dev)
        ps = f.sum(0)
        zero = torch.zeros_like(ps)
        F, u0 = [zero] * 3, [zero] * 3
        for a in dim:
            F[a] = mu * g[a] + rep[a] - ps / 3.0 * dr * g[a] + (rho - self.rho_bar) * p["g"][a]
            u0[a] = F[a] / (2.0 * rho) + sum(c[a] * fi for c, fi in zip(self.c, f) if c[a])
        M = {(a, b): sum(c[a] * c[b] * fi for c, fi in zip(self.c, f) if c[a] * c[b]) - (ps / 3.0 if a == b else 0.0)
             for a in dim for b in dim if a <= b}
        ab = lambda a, b: (min(a, b), max(a, b))  # noqa: E731
        u = [zero] * 3
        for a in dim:
            Fn = -3.0 * nu * om * sum((M[ab(a, b)] - u0[a] * u0[b]) * dr * g[b] for b in dim)
            u[a] = u0[a] + Fn / (2.0 * rho)
            F[a] = (F[a] + Fn) / rho
        if post:
            A = {k: M[k] - u[k[0]] * u[k[1]] + 0.5 * (u[k[0]] * F[k[1]] + u[k[1]] * F[k[0]]) for k in M}
            tr = sum(A[a, a] for a in dim)
            uu, uF = sum(x * x for x in u), sum(x * y for x, y in zip(u, F))
            Au = [sum(A[ab(a, b)] * u[b] for b in dim) for a in dim]
            k = 1.0 - om
            even = ps - 1.5 * uu - 1.5 * k * tr - 1.5 * uF
            odd = 3.0 - 4.5 * uu - 4.5 * k * tr
            for i, (c, w) in enumerate(zip(self.c, self.w)):
                cu, cF = sum((c[a] * u[a] for a in dim), zero), sum((c[a] * F[a] for a in dim), zero)
                cA = sum((c[a] * c[b] * A[ab(a, b)] for a in dim for b in dim if c[a] * c[b]), zero)
                v = even + 4.5 * cu * (cu + cF) + 4.5 * k * cA + cu * (odd + 4.5 * cu * cu + 13.5 * k * cA)
                v = v + 1.5 * cF - 9.0 * k * sum((c[a] * Au[a] for a in dim), zero)
                f[i] = torch.roll(w * v, (c[2], c[1], c[0]), (0, 1, 2))
        return u, ps

    def advance(self, phi, u):
        p = self.p
        kappa = 4.0 * p["D"] / p["eps"]
        n = self.normal(self.grad(phi))
        new = phi + p["D"] * 6.0 * (self.smooth(phi) - phi)
        for a in range(self.dim):
            new -= kappa * self.d(phi * (1.0 - phi) * n[a], a)
            up = self.at(phi, a, 1) - phi
            dn = self.at(up, a, -1)
            slope = torch.where(up * dn > 0.0, torch.where(up.abs() < dn.abs(), up, dn), torch.zeros_like(up))
            uf = 0.5 * (u[a] + self.at(u[a], a, 1))
            flux = uf * torch.where(uf >= 0.0, phi + 0.5 * slope, self.at(phi - 0.5 * slope, a, 1))
            new -= flux - self.at(flux, a, -1)
        return new

    def film(self, phi):
        g = self.grad(phi)
        F, i = self.repulsion(phi, g)
        if not len(i):
            return [0.0] * 7
        n = self.normal(g)
        Fn = sum(F[a] * n[a] for a in range(3)).reshape(-1)[i].abs().sum()
        cn = (self.chemical(phi) * sum(g[a] * n[a] for a in range(3))).reshape(-1)[i].abs().sum()
        s = torch.sqrt((F * F).sum(0)).reshape(-1)[i]
        v = [float(len(i)), float(Fn), float(cn), float(s.max()), float(s.sum())]
        return v + [v[1] / v[2], v[4] / v[0]]

    def run(self, steps, every=0):
        p = self.p
        phi, u = (t.reshape((-1,) + self.shape) for t in _fields(p, self.dev))
        phi = phi[0]
        self.rho_bar = float((p["rho_g"] + (p["rho_l"] - p["rho_g"]) * phi).mean())
        f = torch.empty((len(self.c),) + self.shape, dtype=torch.float64, device=self.dev)
        uu = (u * u).sum(0)
        for i, (c, w) in enumerate(zip(self.c, self.w)):
            cu = sum((c[a] * u[a] for a in range(self.dim)), torch.zeros_like(uu))
            f[i] = w * (cu * (3.0 - 4.5 * uu) + 4.5 * cu * cu - 1.5 * uu + 4.5 * cu ** 3)
        films = []
        for n in range(steps):
            u, _ = self.hydro(f, phi, True)
            phi = self.advance(phi, u)
            if every and (n + 1) % every == 0:
                films.append(self.film(phi))
        u, ps = self.hydro(f, phi, False)
        return phi.reshape(-1), torch.stack(u).reshape(-1), ps.reshape(-1), films


def exact(case, seed):
    if work(case)["bytes"] > 4.0e11:  # too long in 64 bits
        return None
    films = case["kind"] == "films"
    got = [_Exact(c, _dev()).run(case["steps"], 20 if films else 0) for c in _configs(case, seed)]
    out = dict(phi=torch.cat([g[0] for g in got]), u=torch.cat([g[1] for g in got]),
               pstar=torch.cat([g[2] for g in got]))
    if films:
        # the counts of film cells turn on comparisons that 32 and 64 bits take differently
        out["films"] = None
    return out
