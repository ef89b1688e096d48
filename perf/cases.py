"""Timed workloads of the library: what its users run, through the public entry points.

A pass advances a lattice (or a batch of lattices) by a number of steps and reads the fields back
on the device, or evaluates the gradient of a drop objective.  The sizes are those of this
repository's scenarios, tests and benchmark; draw() spreads over the ranges between them.

exact() restates the method (D2Q9, chemical-potential or pseudopotential force, curved boundary
links with mass compensation) in plain 64-bit torch, without the library, and takes gradients with
torch's automatic differentiation.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2203_04508_gb300 as G

# equation of state, collision and boundary constants of every scene (mesh scaling k, gradient
# coefficient kappa, interface width): the values the repository's scenarios use
K_MESH, KAPPA, WIDTH = 0.25, 0.05, 5.0
PR = dict(eos=G.EOS_PR, a=2 / 49, b=2 / 21, R=1.0, omega=0.344, T_over_Tc=0.7, kappa=0.01)


# ---------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # a parameter study's smallest lattice: ragged in both directions, two cylinders of
        # opposite wettability; the step is a chain of small kernels
        dict(name="drops_131x97", kind="lattice", scene="array", nx=131, ny=97, n_cyl=2, steps=25),
        # the verification set-up: 64-bit populations, single relaxation time, neutral cylinder
        dict(name="fp64_bgk_128x128", kind="lattice", scene="cylinder", nx=128, ny=128, fp64=True, bgk=True, steps=25),
        # a drop spreading on a flat substrate cut between the nodes, Peng-Robinson
        dict(name="flat_pr_500x300", kind="lattice", scene="flat", nx=500, ny=300, pr=True, steps=50),
        # a drop falling onto a cylinder, the film-thickness study's lattice
        dict(name="impact_600x1200", kind="lattice", scene="impact", nx=600, ny=1200, steps=50),
        # sixteen drops on sixteen cylinders: both population lattices fit in the L2 cache
        dict(name="drops_1024x1024", kind="lattice", scene="array", nx=1024, ny=1024, n_cyl=16, steps=40),
        # drop impact on the largest lattice (the benchmark's)
        dict(name="impact_2048x4096", kind="lattice", scene="impact", nx=2048, ny=4096, steps=20),
        # the same with the pseudopotential force
        dict(name="pseudo_2048x4096", kind="lattice", scene="impact", nx=2048, ny=4096, pseudo=True, steps=20),
        # the same in one population lattice, updated in place (the memory-saving layout)
        dict(name="one_lattice_2048x4096", kind="lattice", scene="impact", nx=2048, ny=4096, aa=True, steps=20),
        # a sweep over sizes, temperatures and contact angles advanced together
        dict(name="batch_64_of_128_768", kind="batch", n=64, nmin=128, nmax=768, steps=50),
        # a sweep of lattices each far too small to fill the device
        dict(name="batch_256_of_64_128", kind="batch", n=256, nmin=64, nmax=128, steps=200),
        # one gradient of the drop objective with respect to wettability, cylinder centre and
        # initial state: checkpointed forward pass and reverse sweep
        dict(name="gradient_512x512", kind="gradient", scene="cylinder", nx=512, ny=512, steps=100),
        # one iteration of a design loop through torch's autograd: a new lattice is set up from
        # the parameters, stepped and swept back
        dict(name="rollout_192x160", kind="rollout", scene="cylinder", nx=192, ny=160, steps=36),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    u = rng.random()
    if u < 0.6:
        scene = rng.choice(["cylinder", "impact", "array", "flat"])
        nx = _log_int(rng, 96, 2304)
        ny = _log_int(rng, max(96, nx // 3), max(97, min(4096, 3 * nx)))
        if scene == "impact":   # room for a drop of a third of the cylinder's radius above it
            nx = max(nx, 160 + nx % 7)
            ny = max(ny, nx + 16)
        c = dict(kind="lattice", scene=scene, nx=nx, ny=ny)
        if scene == "array":
            # as many cylinders as leave each a cell of about 64 x 64
            c["n_cyl"] = rng.randint(1, max(1, min(12, (nx // 64) * (ny // 64))))
        if scene == "cylinder" and rng.random() < 0.3:
            c["periodic"] = True
        v = rng.random()
        if scene == "flat":
            c["pr"] = True
        elif v < 0.15:
            c["pseudo"] = True
        elif v < 0.30:
            c["aa"] = True
        elif v < 0.45:
            c["fp64"] = True
            c["bgk"] = rng.random() < 0.5
        top = 1.6e7 if c.get("fp64") else 1.6e8   # node updates a pass
        c["steps"] = max(1, min(_log_int(rng, 4, 60), int(top / (nx * ny))))
        return c
    if u < 0.8:
        nmin = _log_int(rng, 64, 256)
        nmax = min(768, _log_int(rng, nmin + 8, 3 * nmin))
        mean = (nmin * nmin + nmin * nmax + nmax * nmax) / 3.0
        n = max(4, min(_log_int(rng, 8, 256), int(1.6e7 / mean)))
        return dict(kind="batch", n=n, nmin=nmin, nmax=nmax, steps=rng.randint(20, 60))
    if u < 0.93:
        return dict(kind="gradient", scene=rng.choice(["cylinder", "impact"]), nx=_log_int(rng, 160, 480),
                    ny=_log_int(rng, 481, 560), steps=rng.randint(20, 90))
    return dict(kind="rollout", scene="cylinder", nx=_log_int(rng, 96, 320), ny=_log_int(rng, 96, 320),
                steps=rng.randint(9, 49))


# ---------------------------------------------------------------------------------------
# scenes: physics and drops from the case and the seed
# ---------------------------------------------------------------------------------------
def _fraction(rng):
    """A sub-lattice offset away from the nodes and from half way between them."""
    f = rng.uniform(0.08, 0.42)
    return f if rng.random() < 0.5 else f + 0.5


def _physics(case, nx, ny):
    p = dict(nx=nx, ny=ny, walls=0 if case.get("periodic") else 1, y_bottom=1.5, y_top=ny - 2.5, eos=G.EOS_CS, a=1.0,
             b=4.0, R=1.0, T_over_Tc=0.6, omega=0.344, k=K_MESH, kappa=KAPPA, coll=G.COLL_MRT, tau=0.8, s_e=1.64,
             s_eps=1.54, s_q=1.7, s_nu=1.0 / 0.8, gx=0.0, gy=0.0, bc=G.BC_PRESENT, cx=[], cy=[], r=[], dmu_w=[],
             dmu_w_walls=0.0, force_model=0)
    if case.get("pr"):
        p.update(PR)
    if case.get("bgk"):
        p.update(coll=G.COLL_BGK, tau=1.0, s_nu=1.0, T_over_Tc=0.7)
    if case.get("pseudo"):
        p.update(force_model=1, T_over_Tc=0.7, k=1.0)
    return p


def _scene(case, seed):
    """(physics, drops) of one lattice."""
    rng = np.random.default_rng([int(seed), 2203])
    nx, ny = int(case["nx"]), int(case["ny"])
    p = _physics(case, nx, ny)
    d = dict(x0=[], y0=[], r0=[], ux0=[], uy0=[], width=WIDTH)
    wet = lambda: 0.0 if case.get("bgk") else float(rng.uniform(-0.15, 0.15) if case.get("pseudo") else rng.uniform(-0.06, 0.06))  # noqa: E731

    def drop(x, y, r, vy=0.0):
        d["x0"].append(float(x)); d["y0"].append(float(y)); d["r0"].append(float(r))
        d["ux0"].append(0.0); d["uy0"].append(float(vy))

    def cylinder(x, y, r):
        p["cx"].append(float(x)); p["cy"].append(float(y)); p["r"].append(float(r)); p["dmu_w"].append(wet())

    scene = case["scene"]
    s = float(min(nx, ny))
    if scene == "flat":
        # the wall line cuts the first fluid row's links at q; a drop resting on it
        q = float(rng.uniform(0.15, 0.95))
        p["y_bottom"] = 2.0 - q
        p["dmu_w_walls"] = float(rng.uniform(-0.04, 0.04))
        r0 = s * float(rng.uniform(0.14, 0.18))
        drop(nx * rng.uniform(0.4, 0.6), p["y_bottom"] + 0.5 * r0, r0)
    elif scene == "cylinder":
        rc = s * float(rng.uniform(0.14, 0.18))
        cx, cy = nx // 2 + _fraction(rng), int(0.3 * ny) + _fraction(rng)
        cylinder(cx, cy, rc)
        drop(cx, cy + rc, 0.6 * rc)
    elif scene == "impact":
        rc = nx * float(rng.uniform(0.14, 0.15))
        cx, cy = nx // 2 + _fraction(rng), int(rc + 6 + nx * 0.005) + _fraction(rng)
        rd = rc / 3.0
        p["gy"] = -1e-6
        cylinder(cx, cy, rc)
        drop(cx, cy + rc + rd + 0.25 * rc, rd, -0.05 if not case.get("pseudo") else -0.02)
    else:
        # cylinders in the cells of a grid, each with a drop on top
        n = int(case["n_cyl"])
        gx = max(1, int(round(math.sqrt(n * nx / ny))))
        gy = -(-n // gx)
        w, h = (nx - 12.0) / gx, (ny - 12.0) / gy
        for k in range(n):
            # a cylinder of radius r and its drop of radius 0.7 r take 3.4 r of the cell's height
            r = min(w / 2.5, h / 4.0) * float(rng.uniform(0.75, 0.95))
            x0, y0 = 6 + w * (k % gx), 6 + h * (k // gx)
            cx = int(x0 + 0.5 * w) + _fraction(rng)
            cy = int(y0 + 1.25 * r + 1.0) + _fraction(rng)
            cylinder(cx, cy, r)
            drop(cx, cy + r, 0.7 * r)
    return p, d


def _batch_scenes(case, seed):
    rng = np.random.default_rng([int(seed), 4])
    # the sizes belong to the case, the rest to the seed
    sizes = np.random.default_rng([int(case["n"]), int(case["nmin"]), int(case["nmax"])]).integers(
        int(case["nmin"]), int(case["nmax"]) + 1, int(case["n"]))
    out = []
    for N in (int(v) for v in sizes):
        p = _physics({}, N, N)
        rc = N * float(rng.uniform(0.15, 0.28))
        rd = min(rc * float(rng.uniform(0.5, 1.0)), (N - 2 * rc - 20) / 2.0)
        cx, cy = N // 2 + _fraction(rng), int(4 + rc) + _fraction(rng)
        p["T_over_Tc"] = float(rng.uniform(0.6, 0.8))
        p["cx"], p["cy"], p["r"], p["dmu_w"] = [cx], [cy], [rc], [float(rng.uniform(-0.06, 0.06))]
        out.append((p, dict(x0=[cx], y0=[cy + rc], r0=[rd], ux0=[0.0], uy0=[0.0], width=WIDTH)))
    return out


def _sizes(case):
    """Nodes of the case's lattices."""
    if case["kind"] != "batch":
        return float(case["nx"]) * case["ny"]
    return float(sum(p["nx"] * p["ny"] for p, _ in _batch_scenes(case, 0)))


# ---------------------------------------------------------------------------------------
# the timed calls
# ---------------------------------------------------------------------------------------
def prepare(case, seed):
    n = int(case["steps"])
    if case["kind"] == "batch":
        scenes = _batch_scenes(case, seed)
        b = G.Batch([p for p, _ in scenes])
        b.set_schedule(1)   # what the autotuner picks for such mixes
        b.init([d for _, d in scenes])
        return dict(kind="batch", b=b, steps=n)
    p, d = _scene(case, seed)
    if case["kind"] == "rollout":
        y = torch.arange(p["ny"], device="cuda", dtype=torch.float32)[:, None]
        params = torch.tensor(G.params_vector(p), dtype=torch.float32, device="cuda")
        return dict(kind="rollout", p=p, d=d, y=y, params=params, steps=n)
    lat = G.Lattice(p, precision=G.LBM_FP64 if case.get("fp64") else G.LBM_FP32,
                    layout=G.LBM_LAYOUT_AA if case.get("aa") else G.LBM_LAYOUT_AB)
    lat.init_droplets(d)
    if case["kind"] == "gradient":
        return dict(kind="gradient", lat=lat, d=d, steps=n)
    lat.prepare_steps(n)
    return dict(kind="lattice", lat=lat, steps=n)


def run(state):
    n = state["steps"]
    if state["kind"] == "lattice":
        state["lat"].step(n)
        rho, vx, vy = state["lat"].fields(on_device=True)
        return dict(rho=rho, vx=vx, vy=vy)
    if state["kind"] == "batch":
        state["b"].step(n)
        out = [inst.fields(on_device=True) for inst in state["b"].instances]
        return {k: torch.cat([o[i].reshape(-1) for o in out]) for i, k in enumerate(("rho", "vx", "vy"))}
    if state["kind"] == "gradient":
        lat = state["lat"]
        lat.init_droplets(state["d"])
        lat.forward_checkpointed(n)
        J, seed = lat.objective(0, seed=True)
        grad, df0 = lat.adjoint(drho=seed, want_df0=True)
        return dict(J=J, grad=grad.astype(np.float32), df0=df0, rho=lat.fields(on_device=True)[0])
    params = state["params"].clone().requires_grad_(True)
    rho = G.rollout(params, state["p"], state["d"], n)
    J = (rho * state["y"]).sum() / rho.sum()   # height of the centre of mass
    J.backward()
    return dict(J=J.detach(), rho=rho.detach(), grad=params.grad)


def work(case):
    """One pass: each step reads and writes the nine populations of every node (about 300
    operations a node); the reverse sweep recomputes the steps, and reads the populations and
    reads and writes their nine adjoints."""
    sz = 8.0 if case.get("fp64") else 4.0
    nodes, n = _sizes(case), float(case["steps"])
    if case["kind"] in ("gradient", "rollout"):
        return dict(bytes=nodes * sz * (n * (18 + 18 + 27) + 12), flops=nodes * n * 1000.0)
    return dict(bytes=nodes * sz * (n * 18 + 3), flops=nodes * n * 300.0)


# ---------------------------------------------------------------------------------------
# the method in 64 bits, plain torch
# ---------------------------------------------------------------------------------------
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
W9 = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
SQ2 = math.sqrt(2.0)


def _pressure(p, RT, aal, r):
    if p["eos"] == G.EOS_CS:
        e = p["b"] * r / 4
        return r * RT * (1 + e + e * e - e ** 3) / (1 - e) ** 3 - p["a"] * r * r
    x = p["b"] * r
    return r * RT / (1 - x) - aal * r * r / (1 + 2 * x - x * x)


def _psi_prime(p, RT, aal, r, log):
    """Bulk chemical potential."""
    if p["eos"] == G.EOS_CS:
        e = p["b"] * r / 4
        return RT * (log(r) + (8 * e - 9 * e * e + 3 * e ** 3) / (1 - e) ** 3) - 2 * p["a"] * r
    x = p["b"] * r
    return (RT * log(r / (1 - x)) - aal / (2 * SQ2 * p["b"]) * log((SQ2 - 1 + x) / (SQ2 + 1 - x)) + RT / (1 - x)
            - aal * r / (1 + 2 * x - x * x))


def _bisect(f, lo, hi):
    at_lo = f(lo) > 0
    for _ in range(200):
        m = 0.5 * (lo + hi)
        if (f(m) > 0) == at_lo:
            lo = m
        else:
            hi = m
    return 0.5 * (lo + hi)


def _coexistence(p):
    """RT, a alpha, gas and liquid density and chemical potential at saturation: the critical
    point from A' B'' = A'' B' of the reduced pressure RT A(s) - a B(s), then equal pressure and
    chemical potential of both phases."""
    if p["eos"] == G.EOS_CS:
        A1 = lambda s: (1 + 4 * s + 4 * s * s - 4 * s ** 3 + s ** 4) / (1 - s) ** 4        # noqa: E731
        A2 = lambda s: (8 + 20 * s - 4 * s * s) / (1 - s) ** 5                             # noqa: E731
        B1, B2, c1, c2, top = (lambda s: 2 * s), (lambda s: 2.0), 4 / p["b"], 16 / p["b"] ** 2, 0.4
    else:
        D = lambda s: 1 + 2 * s - s * s                                                    # noqa: E731
        A1 = lambda s: 1 / (1 - s) ** 2                                                    # noqa: E731
        A2 = lambda s: 2 / (1 - s) ** 3                                                    # noqa: E731
        B1 = lambda s: (2 * s + 2 * s * s) / D(s) ** 2                                     # noqa: E731
        B2 = lambda s: ((2 + 4 * s) * D(s) - 2 * (2 * s + 2 * s * s) * (2 - 2 * s)) / D(s) ** 3  # noqa: E731
        c1, c2, top = 1 / p["b"], 1 / p["b"] ** 2, 0.6
    sc = _bisect(lambda s: A1(s) * B2(s) - A2(s) * B1(s), 0.02, top)
    RT = p["T_over_Tc"] * p["a"] * c2 / c1 * B1(sc) / A1(sc)
    aal = p["a"]
    if p["eos"] == G.EOS_PR:
        kw = 0.37464 + 1.54226 * p["omega"] - 0.26992 * p["omega"] ** 2
        aal *= (1 + kw * (1 - math.sqrt(p["T_over_Tc"]))) ** 2
    P = lambda r: _pressure(p, RT, aal, r)                       # noqa: E731
    mu = lambda r: _psi_prime(p, RT, aal, r, math.log)           # noqa: E731
    # the pressure's local maximum and minimum on either side of the critical density (reduced
    # density 1: close packing), and the densities of pressure ps on the two stable branches
    dP = lambda s: A1(s) * RT - (aal * c2 / c1) * B1(s)          # noqa: E731
    s1, s2 = c1 * _bisect(dP, 1e-9, sc), c1 * _bisect(dP, sc, 0.999)
    gas = lambda ps: _bisect(lambda r: P(r) - ps, 1e-300, s1)               # noqa: E731
    liq = lambda ps: _bisect(lambda r: P(r) - ps, s2, c1 * (1 - 1e-12))     # noqa: E731
    ps = _bisect(lambda q: mu(gas(q)) - mu(liq(q)), max(P(s2), P(s1) * 1e-9), P(s1))
    rg, rl = gas(ps), liq(ps)
    return RT, aal, rg, rl, mu(rg)


def _mrt_matrix(p):
    """M^-1 (I - S) M, acting on the non-equilibrium populations."""
    M = np.array([[1, 1, 1, 1, 1, 1, 1, 1, 1], [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
                  [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
                  [0, 0, -2, 0, 2, 1, 1, -1, -1], [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]], float)
    S = np.diag([0, p["s_e"], p["s_eps"], 0, p["s_q"], 0, p["s_q"], p["s_nu"], p["s_nu"]])
    return np.linalg.inv(M) @ (np.eye(9) - S) @ M


class _Exact:
    """One lattice in 64 bits.  dmu, dmu_walls, cx, cy may be tensors that require gradients."""

    def __init__(self, p, dmu=None, dmu_walls=None, cx=None, cy=None):
        dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        t = lambda v: torch.as_tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
        self.p, self.dev = p, dev
        self.RT, self.aal, self.rg, self.rl, self.mu_sat = _coexistence(p)
        n = len(p["r"])
        cx = t(p["cx"]) if cx is None else cx
        cy = t(p["cy"]) if cy is None else cy
        dmu = t(p["dmu_w"]) if dmu is None else dmu
        dmu_walls = t(p["dmu_w_walls"]) if dmu_walls is None else dmu_walls
        X = torch.arange(p["nx"], device=dev, dtype=torch.float64)[None, :].expand(p["ny"], -1)
        Y = torch.arange(p["ny"], device=dev, dtype=torch.float64)[:, None].expand(-1, p["nx"])
        self.X, self.Y = X, Y
        body = torch.full((p["ny"], p["nx"]), -1, device=dev, dtype=torch.int64)
        inside = [(X - float(p["cx"][b])) ** 2 + (Y - float(p["cy"][b])) ** 2 <= p["r"][b] ** 2 for b in range(n)]
        if p["walls"]:
            inside += [Y <= p["y_bottom"], Y >= p["y_top"]]
        for b in reversed(range(len(inside))):
            body[inside[b]] = b
        self.fluid = body < 0
        fl = self.fluid
        near = lambda m: torch.stack([self.at(m, i) for i in range(1, 9)])  # noqa: E731
        self.s1 = ~fl & near(fl).any(0)
        self.s2 = ~fl & ~self.s1 & near(self.s1).any(0)
        w = t(W9[1:])[:, None, None]
        self.w1 = near(fl) * w * self.s1
        self.w2 = near(self.s1) * w * self.s2
        self.w1, self.w2 = (m / m.sum(0).clamp_min(1e-300) for m in (self.w1, self.w2))
        # wall chemical potential (or the pseudopotential's wall factor) of the solid layers
        vals = torch.cat([dmu, dmu_walls.reshape(1)])
        layer = (self.s1 | self.s2)
        self.wall = torch.where(layer, vals[body.clamp(0, n)], torch.zeros_like(X)) if n or p["walls"] else torch.zeros_like(X)
        # cut links: per direction the fluid nodes with a solid neighbour, and the fraction q
        self.links = []
        for i in range(1, 9):
            y1, x1 = torch.nonzero(fl & ~self.at(fl, i), as_tuple=True)
            if not len(x1):
                continue
            xs, ys = (x1 + EX[i]) % p["nx"], (y1 + EY[i]) % p["ny"]
            q = torch.full((len(x1),), math.inf, device=dev, dtype=torch.float64)
            xf, yf = x1.double(), y1.double()
            for b, m in enumerate(inside):
                if b < n:
                    dx, dy = xf - cx[b], yf - cy[b]
                    A, B = float(EX[i] ** 2 + EY[i] ** 2), 2 * (dx * EX[i] + dy * EY[i])
                    C = dx * dx + dy * dy - p["r"][b] ** 2
                    ok = m[ys, xs]
                    disc = torch.where(ok, B * B - 4 * A * C, torch.ones_like(B))
                    qb = (-B - torch.sqrt(disc)) / (2 * A)
                else:
                    ok = m[ys, xs]
                    qb = yf - p["y_bottom"] if b == n else p["y_top"] - yf
                q = torch.where(ok & (qb < q), qb, q)
            x2f = self.at(fl, OPP[i])[y1, x1]
            self.links.append((i, y1, x1, q, x2f))
        if p["coll"] == G.COLL_MRT:
            self.relax = t(_mrt_matrix(p))
        else:
            self.relax = t((1 - 1 / p["tau"]) * np.eye(9))
        self.e = t([EX, EY])
        self.w = t(W9)[:, None, None]

    @staticmethod
    def at(v, i):
        """v at x + e_i."""
        return torch.roll(v, (-EY[i], -EX[i]), (-2, -1))

    def feq(self, r, ux, uy):
        eu = self.e[0][:, None, None] * ux + self.e[1][:, None, None] * uy
        return self.w * r * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))

    def init(self, d):
        phi = torch.zeros_like(self.X)
        ux, uy = torch.zeros_like(phi), torch.zeros_like(phi)
        for x0, y0, r0, u0, v0 in zip(d["x0"], d["y0"], d["r0"], d["ux0"], d["uy0"]):
            ph = 0.5 - 0.5 * torch.tanh(2 * (torch.sqrt((self.X - x0) ** 2 + (self.Y - y0) ** 2) - r0) / d["width"])
            m = ph > phi
            phi, ux, uy = torch.where(m, ph, phi), torch.where(m, u0 * ph, ux), torch.where(m, v0 * ph, uy)
        r = 0.5 * (self.rg + self.rl) + 0.5 * (self.rg - self.rl) * (1 - 2 * phi)
        return torch.where(self.fluid, self.feq(r, ux, uy), torch.zeros_like(phi))

    def state(self, f):
        """Density (solid layers filled), momentum and force."""
        p, fl = self.p, self.fluid
        r = torch.where(fl, f.sum(0), torch.full_like(f[0], self.rg))
        jx, jy = ((f * self.e[k][:, None, None]).sum(0) for k in (0, 1))
        rs = torch.where(fl, r, torch.zeros_like(r))
        for w in (self.w1, self.w2):
            rs = rs + sum(w[i - 1] * self.at(rs, i) for i in range(1, 9))
        if p["force_model"]:
            ok = fl | self.s1 | self.s2
            psi = torch.sqrt((2 * (rs / 3 - p["k"] ** 2 * _pressure(p, self.RT, self.aal, rs))).clamp_min(0))
            psi = torch.where(ok, psi * (1 + self.wall), torch.zeros_like(psi))
            g = [sum((1 / 3 if i < 5 else 1 / 12) * self.at(psi, i) * e[i] for i in range(1, 9) if e[i]) for e in (EX, EY)]
            Fx, Fy = r * p["gx"] + psi * g[0], r * p["gy"] + psi * g[1]
        else:
            s = lambda v, a, k: torch.roll(v, -k, a)  # noqa: E731
            lap = sum(16 * (s(rs, a, 1) + s(rs, a, -1)) - s(rs, a, 2) - s(rs, a, -2) - 30 * rs for a in (0, 1)) / 12
            mu = p["k"] ** 2 * (_psi_prime(p, self.RT, self.aal, r, torch.log) - self.mu_sat) - p["kappa"] * lap
            mu = torch.where(fl, mu, self.wall)
            grad = lambda v, a: (8 * (s(v, a, 1) - s(v, a, -1)) - (s(v, a, 2) - s(v, a, -2))) / 12  # noqa: E731
            Fx = r * p["gx"] - r * grad(mu, 1) + grad(rs, 1) / 3
            Fy = r * p["gy"] - r * grad(mu, 0) + grad(rs, 0) / 3
        z = torch.zeros_like(r)
        return r, jx, jy, torch.where(fl, Fx, z), torch.where(fl, Fy, z)

    def step(self, f):
        r, jx, jy, Fx, Fy = self.state(f)
        ux, uy = jx / r, jy / r
        eq = self.feq(r, ux, uy)
        eq2 = self.feq(r, ux + Fx / r, uy + Fy / r)
        post = eq2 + (self.relax @ (f - eq).reshape(9, -1)).reshape(f.shape)
        post = torch.where(self.fluid, post, torch.zeros_like(post))
        new = torch.stack([torch.roll(post[i], (EY[i], EX[i]), (0, 1)) for i in range(9)])
        edm = eq2 - eq
        ny, nx = self.X.shape
        comp = torch.zeros_like(r)
        vals, idx = [], []
        for i, y1, x1, q, x2f in self.links:
            a, c, Fi = post[i][y1, x1], post[OPP[i]][y1, x1], edm[i][y1, x1]
            b2 = post[i][(y1 - EY[i]) % ny, (x1 - EX[i]) % nx]
            low = torch.where(x2f, 2 * q * a + (1 - 2 * q) * (b2 + Fi), a)
            v = torch.where(q < 0.5, low, (a + (2 * q - 1) * (c + Fi)) / (2 * q))
            vals.append(v)
            idx.append((OPP[i] * ny + y1) * nx + x1)
            comp = comp.index_put((y1, x1), a - v, accumulate=True)
        if vals:
            new = new.reshape(-1).index_put((torch.cat(idx),), torch.cat(vals)).reshape(new.shape)
        return torch.cat([(new[0] + comp)[None], new[1:]])

    def fields(self, f):
        r, jx, jy, Fx, Fy = self.state(f)
        z = torch.zeros_like(r)
        return [torch.where(self.fluid, v, z) for v in (r, (jx + 0.5 * Fx) / r, (jy + 0.5 * Fy) / r)]

    def objective(self, r, b):
        """Centre-of-mass height of the excess density plus the wetted arc of cylinder b."""
        ex = torch.where(self.fluid, r - self.rg, torch.zeros_like(r))
        inside = (self.X - float(self.p["cx"][b])) ** 2 + (self.Y - float(self.p["cy"][b])) ** 2 <= self.p["r"][b] ** 2
        touch = self.fluid & torch.stack([self.at(inside, i) for i in range(1, 9)]).any(0)
        arc = 2 * math.pi * self.p["r"][b] / touch.sum()
        return (ex * self.Y).sum() / ex.sum() + arc * (ex * touch).sum() / (self.rl - self.rg)


def _rolled(L, f, n):
    """n steps with the states kept every few steps only, for the gradient."""
    from torch.utils.checkpoint import checkpoint

    def some(f, k):
        for _ in range(k):
            f = L.step(f)
        return f
    k = max(1, int(math.sqrt(n)))
    for s in range(0, n, k):
        f = checkpoint(some, f, min(k, n - s), use_reentrant=False)
    return f


def exact(case, seed):
    n = int(case["steps"])
    # about 0.4 ms a step of launches, and 60 ns a thousand nodes
    cost = n * (4e-3 * (case["n"] if case["kind"] == "batch" else 1) + 6e-9 * _sizes(case))
    if case["kind"] in ("gradient", "rollout"):
        cost *= 4
    if cost > 20:
        return None
    if case["kind"] == "batch":
        out = []
        with torch.no_grad():
            for p, d in _batch_scenes(case, seed):
                L = _Exact(p)
                f = L.init(d)
                for _ in range(n):
                    f = L.step(f)
                out.append([v.reshape(-1) for v in L.fields(f)])
        return {k: torch.cat([o[i] for o in out]) for i, k in enumerate(("rho", "vx", "vy"))}
    p, d = _scene(case, seed)
    if case["kind"] == "lattice":
        with torch.no_grad():
            L = _Exact(p)
            f = L.init(d)
            for _ in range(n):
                f = L.step(f)
            return dict(zip(("rho", "vx", "vy"), L.fields(f)))
    m = len(p["r"])
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    leaf = G.params_vector(p)
    if case["kind"] == "rollout":
        leaf = leaf.astype(np.float32)   # as the caller hands them over
        p = G.with_params(p, leaf)
    leaf = torch.tensor(leaf, dtype=torch.float64, device=dev, requires_grad=True)
    L = _Exact(p, leaf[:m], leaf[m], leaf[m + 1::2], leaf[m + 2::2])
    f0 = L.init(d).detach().requires_grad_(True)
    r = _rolled(L, f0, n).sum(0)
    rho = torch.where(L.fluid, r, torch.zeros_like(r))
    if case["kind"] == "rollout":
        J = (rho * L.Y).sum() / rho.sum()
        J.backward()
        return dict(J=J.detach(), rho=rho.detach(), grad=leaf.grad)
    J = L.objective(r, 0)
    J.backward()
    return dict(J=J.detach(), grad=leaf.grad, df0=torch.where(L.fluid, f0.grad, torch.zeros_like(r)),
                rho=rho.detach())
