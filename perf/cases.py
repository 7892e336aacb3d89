"""Measured cases: what a user of this framework has it do.

A pass is a call or two of the Python layer as the quick start and the
examples make them: a number of iterations on a bound solver and the read of
the fields, a whole steady solve, a state handed over and taken back, an
adjoint.  The library's default launch shapes are used throughout.

Outputs are held to the precision they are computed in: mixed-precision
solvers store and sweep f in float32, so their results are returned as
float32; float64 solvers return float64.

exact() is an independent float64 statement of the scheme (Section 2 of the
paper) on plain cell and face lists in torch, structured and unstructured
alike; it shares only the problem descriptions (meshes, gas, boundaries).
"""
import math

import numpy as np
import torch

from paper_1709_01819_gb300 import inputs as I
from paper_1709_01819_gb300.solver import BatchSolver, Solver


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # the smallest call: a 1-D Couette flow solved from rest to 1e-6, wall
        # quantities read (latency and launches; the periodic direction is one cell wide)
        {"name": "couette64_solve", "kind": "solve", "flow": "couette", "n": 64, "m": 1, "nv": 32, "rule": "trap",
         "prec": "mixed", "Kn": 0.1, "cfl": 100.0, "iters": 2000, "tol": 1e-6},
        # the headline workload: lid-driven cavity, Shakhov, trapezoid velocities
        {"name": "cavity64", "kind": "iterate", "flow": "cavity", "n": 64, "m": 64, "nv": 32, "rule": "trap",
         "prec": "mixed", "Kn": 0.075, "cfl": 1000.0, "iters": 32},
        # the same in float64, the precision results are validated in
        {"name": "cavity64_fp64", "kind": "iterate", "flow": "cavity", "n": 64, "m": 64, "nv": 32, "rule": "trap",
         "prec": "fp64", "Kn": 0.075, "cfl": 1000.0, "iters": 4},
        # near-continuum cavity on a stretched grid, Gauss-Hermite velocities
        {"name": "cavity128_gh28", "kind": "iterate", "flow": "cavity", "n": 128, "m": 128, "nv": 28, "rule": "gh",
         "prec": "mixed", "Kn": 1e-3, "cfl": 1e4, "beta": 1.83297, "iters": 16},
        # ragged block, odd velocity count (ties on the faces), point-relaxation predictor
        {"name": "cavity90x70_relax9", "kind": "iterate", "flow": "cavity", "n": 90, "m": 70, "nv": 27,
         "rule": "simpson", "prec": "mixed", "Kn": 0.5, "cfl": 1000.0, "relax": 9, "iters": 16},
        # the largest: hypersonic cylinder, limiter, far field, periodic O-grid; drag and wall loads read
        {"name": "cylinder121x81_v89", "kind": "iterate", "flow": "cylinder", "n": 121, "m": 81, "nv": 89,
         "rule": "simpson", "prec": "mixed", "Kn": 0.1, "Ma": 5.0, "cfl": 30.0, "iters": 4},
        # a parameter study: seeded cavities of several sizes advanced together
        {"name": "batch16", "kind": "batch", "count": 16, "lo": 32, "hi": 96, "nv": 32, "rule": "trap", "prec": "mixed",
         "cfl": 1000.0, "iters": 16},
        # unstructured mesh of triangles (level-scheduled sweeps)
        {"name": "tri64", "kind": "iterate", "flow": "tri", "n": 64, "m": 64, "nv": 32, "rule": "trap",
         "prec": "mixed", "Kn": 0.075, "cfl": 10.0, "iters": 16},
        # explicit DUGKS time steps, the scheme the implicit one is compared with
        {"name": "explicit61", "kind": "iterate", "flow": "cavity", "n": 61, "m": 61, "nv": 32, "rule": "trap",
         "prec": "mixed", "Kn": 0.075, "cfl": 1000.0, "explicit": True, "iters": 32},
        # a coupled program: state in from page-locked host arrays, a few iterations, state out
        {"name": "state48x40", "kind": "state", "flow": "cavity", "n": 48, "m": 40, "nv": 28, "rule": "trap",
         "prec": "mixed", "Kn": 0.2, "cfl": 1000.0, "iters": 16},
        # the backward direction: gradient of the lid force by the discrete adjoint
        {"name": "adjoint24", "kind": "adjoint", "flow": "cavity", "n": 24, "m": 24, "nv": 16, "rule": "trap",
         "prec": "fp64", "Kn": 0.1, "cfl": 1000.0, "iters": 32},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "cavity", "cavity", "cavity", "fp64", "cylinder", "tri", "explicit", "state", "batch",
                       "adjoint"])
    kn = 10.0 ** rng.uniform(-2.0, 1.0)
    rule = rng.choice(["trap", "gh", "simpson"])
    nv = _logint(rng, 16, 40)
    nv += rule == "simpson" and nv % 2 == 0
    base = {"kind": "iterate", "flow": "cavity", "n": _logint(rng, 20, 128), "m": _logint(rng, 20, 128), "nv": nv,
            "rule": rule, "prec": "mixed", "Kn": kn, "cfl": 1000.0, "iters": rng.randrange(4, 33)}
    if kind == "solve":
        return {**base, "kind": "solve", "flow": "couette", "n": _logint(rng, 16, 128), "m": 1, "Kn": max(kn, 0.1),
                "cfl": 100.0, "iters": 1000, "tol": 1e-6}
    if kind == "cavity":
        option = rng.choice(["", "", "beta", "relax", "implicit_wall"])
        if option == "beta":
            return {**base, "m": base["n"], "beta": rng.uniform(0.8, 1.9)}
        return {**base, **({option: rng.choice([1, 4, 9, 16])} if option == "relax" else {option: True} if option else {})}
    if kind == "fp64":
        return {**base, "prec": "fp64", "n": _logint(rng, 16, 64), "m": _logint(rng, 16, 64), "nv": 16 + nv % 17,
                "rule": "trap", "iters": rng.randrange(2, 6)}
    if kind == "cylinder":
        return {**base, "flow": "cylinder", "n": _logint(rng, 24, 121), "m": _logint(rng, 16, 81),
                "nv": 41 + 2 * rng.randrange(0, 25), "rule": "simpson", "Kn": max(kn, 0.05), "Ma": rng.uniform(1.5, 3.0),
                "cfl": 10.0, "iters": rng.randrange(2, 6)}
    if kind == "tri":
        n = _logint(rng, 12, 64)
        return {**base, "flow": "tri", "n": n, "m": n, "cfl": 10.0}
    if kind == "explicit":
        return {**base, "n": _logint(rng, 12, 80), "m": _logint(rng, 12, 80), "explicit": True}
    if kind == "state":
        return {**base, "kind": "state", "n": _logint(rng, 16, 64), "m": _logint(rng, 16, 64)}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randrange(4, 17), "lo": rng.randrange(16, 40), "hi": rng.randrange(48, 97),
                "nv": nv, "rule": rule, "prec": "mixed", "cfl": 1000.0, "iters": rng.choice([8, 16])}
    return {**base, "kind": "adjoint", "prec": "fp64", "n": _logint(rng, 8, 24), "m": _logint(rng, 8, 24),
            "nv": rng.randrange(12, 21), "rule": "trap", "Kn": max(kn, 0.05), "iters": rng.randrange(16, 65)}


# --------------------------------------------------------------------------
# what a user's program has in hand, and one pass
# --------------------------------------------------------------------------

_RULES = {"trap": I.NC_TRAP, "simpson": I.NC_SIMPSON, "gh": I.GAUSS_HERMITE}


def _problem(case, rng):
    """The case's problem; the seed moves the Knudsen number, the wall (or free
    stream) speed and the wall temperature."""
    kn = case.get("Kn", 1.0) * 10.0 ** rng.uniform(-0.1, 0.1)
    speed = rng.uniform(0.8, 1.2)
    tw = rng.uniform(0.95, 1.05)
    nv, cfl = case["nv"], case["cfl"]
    if case["flow"] == "couette":
        p = I.couette(case["n"], 0.1 * speed, kn, nv, 4.0, cfl, Tw=1.0)
    elif case["flow"] == "cylinder":
        ma = case["Ma"]
        p = I.cylinder(case["n"], case["m"], kn, ma * (0.95 + 0.1 * (speed - 0.8) / 0.4), nv,
                       vmax=15.0 if ma > 4 else 9.0, cfl_imp=cfl, Tw=tw)
    elif case["flow"] == "tri":
        p = I.tri_cavity(case["n"], Kn=kn, U=0.15 * speed, nv=nv, cfl_imp=cfl)
    else:
        p = I.cavity(case["n"], kn, 0.15 * speed, nv, 4.0, cfl, stretch_beta=case.get("beta"))
        if case["m"] != case["n"]:
            p.nodes_x, p.nodes_y = I.uniform_nodes(case["n"], case["m"], 0.0, 1.0, 0.0, case["m"] / case["n"])
    if case["flow"] in ("cavity", "tri"):
        west = list(p.bc[I.IMIN])
        west[4] = tw  # a heated side wall
        p.bc[I.IMIN] = tuple(west)
    p.vrule = _RULES[case["rule"]]
    p.relax_sweeps = case.get("relax", 0)
    p.implicit_wall = 1 if case.get("implicit_wall") else 0
    return p


def _problems(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] != "batch":
        return [_problem(case, rng)]
    # sizes are the case's own (not the seed's): the work of a pass does not depend on the seed
    sizes = np.random.default_rng(case["count"] * 1000 + case["lo"]).integers(case["lo"], case["hi"] + 1, case["count"])
    return [_problem({**case, "flow": "cavity", "n": int(n), "m": int(n), "Kn": 10.0 ** rng.uniform(-2.0, 1.0)}, rng)
            for n in sizes]


def _start_state(prob, seed):
    """A smooth non-equilibrium state (G, H, W): per cell a Maxwellian of
    varying density, velocity and temperature times a smooth anisotropy, on the
    solver's velocity nodes."""
    d = _device()
    g = torch.Generator().manual_seed(seed)
    a = (0.05 * (torch.rand(6, generator=g, dtype=torch.float64) - 0.5)).tolist()
    x, y, _ = _velocities(prob)
    x, y = torch.as_tensor(x, device=d), torch.as_tensor(y, device=d)
    j, i = torch.meshgrid(torch.arange(prob.nj, device=d, dtype=torch.float64),
                          torch.arange(prob.ni, device=d, dtype=torch.float64), indexing="ij")
    s, t = ((i + 0.5) / prob.ni).reshape(-1, 1), ((j + 0.5) / prob.nj).reshape(-1, 1)
    rho = 1.0 + 0.1 * torch.sin(2 * math.pi * s + a[0]) * torch.cos(math.pi * t)
    u, v = 0.05 * torch.cos(math.pi * t) + a[1], 0.03 * torch.sin(2 * math.pi * s) + a[2]
    T = 1.0 + 0.05 * torch.cos(math.pi * s) * torch.sin(math.pi * t) + a[3]
    RT = prob.RT_ref * T
    c2 = (x - u) ** 2 + (y - v) ** 2
    G = rho / (2 * math.pi * RT) * torch.exp(-c2 / (2 * RT)) * (1.0 + a[4] * (x - u) * (y - v))
    H = prob.K * RT * G * (1.0 + a[5] * (x - u))
    W = torch.cat([rho, rho * u, rho * v, 0.5 * rho * (u * u + v * v + (prob.K + 2) * RT)], 1)
    return G, H, W


def prepare(case, seed):
    probs = _problems(case, seed)
    if case["kind"] == "batch":
        return {"case": case, "batch": BatchSolver(probs, case["prec"])}
    s = Solver(probs[0], case["prec"], explicit=bool(case.get("explicit")))
    s.init_uniform()
    state = {"case": case, "solver": s}
    if case["kind"] == "state":
        state["host"] = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t).numpy()
                         for t in _start_state(probs[0], seed)]
    if case["kind"] == "adjoint":
        s.iterate(600, 1e-9)  # the adjoint is taken at a converged state
    return state


def _typed(case, v):
    v = np.asarray(v)
    return v.astype(np.float32) if case["prec"] == "mixed" else v


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        b.iterate(case["iters"])
        return [_typed(case, s.moments()) for s in b.solvers]
    s = state["solver"]
    if case["kind"] == "solve":
        s.init_uniform()
        s.iterate(case["iters"], case["tol"])
        return {"moments": _typed(case, s.moments()), "wall": _typed(case, s.wall(I.JMAX))}
    if case["kind"] == "state":
        s.set_state(*state["host"])
        s.iterate(case["iters"])
        G, H, W = s.get_state()
        return {"G": _typed(case, G), "H": _typed(case, H), "W": _typed(case, W)}
    if case["kind"] == "adjoint":
        _, J, grad, _, _ = s.adjoint(0, 1 << I.JMAX, [I.param(I.PAR_KN), I.param(I.PAR_WALL_U, 1 << I.JMAX)],
                                     case["iters"], 0.0, keep_state=True)
        lg, lh, lw = s.adjoint_state(0)
        return {"J": np.float64(J), "grad": np.asarray(grad), "lamG": lg, "lamH": lh, "lamW": lw}
    s.iterate(case["iters"])
    out = {"moments": _typed(case, s.moments())}
    if case["prec"] == "fp64":  # validation runs keep the whole distribution
        out["G"], out["H"], out["W"] = s.get_state()
    if case["flow"] == "cylinder":
        out["wall"] = _typed(case, s.wall(I.JMIN))
        out["drag"] = _typed(case, s.wall_force(1 << I.JMIN))
    return out


def work(case):
    """Per iteration every cell-velocity's pair {G, H} is read and written once
    (an iteration depends on all of the one before through its sweeps); the
    operations are the scheme's own arithmetic: three equilibria, two faces'
    reconstruction and flux, moments and two sweeps per cell-velocity."""
    scalar = 8 if case["prec"] == "fp64" else 4
    if case["kind"] == "batch":
        cells = sum(p.ncells for p in _problems(case, 0))
    else:
        cells = case["n"] * case["m"] * (2 if case["flow"] == "tri" else 1)
    iters = 600 if case["kind"] == "solve" else case["iters"]  # a Couette flow at Kn 0.1 takes about 600
    cv = float(cells) * case["nv"] ** 2
    flops = 900.0 if case["kind"] == "adjoint" else 400.0
    return {"bytes": iters * cv * 4 * scalar + cells * 48.0, "flops": iters * cv * flops}


# --------------------------------------------------------------------------
# the scheme in float64 on cell and face lists
# --------------------------------------------------------------------------

def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _rule(prob, n, lo, hi):
    if prob.vrule == I.GAUSS_HERMITE:
        x, w = np.polynomial.hermite.hermgauss(n)
        unit = math.sqrt(2.0 * prob.RT_ref)
        return unit * x, unit * w * np.exp(x * x)
    x = 0.5 * (lo + hi) + (np.arange(n) - 0.5 * (n - 1)) * ((hi - lo) / (n - 1))
    w = np.full(n, (hi - lo) / (n - 1))
    if prob.vrule == I.NC_TRAP:
        w[[0, -1]] *= 0.5
    else:
        w *= np.where(np.arange(n) % 2 == 1, 4.0, 2.0) / 3.0
        w[[0, -1]] = (hi - lo) / (n - 1) / 3.0
    return x, w


def _velocities(prob):
    x0, x1, y0, y1 = prob.vrange
    x, wx = _rule(prob, prob.nvx, x0, x1)
    y, wy = _rule(prob, prob.nvy, y0, y1)
    return np.tile(x, prob.nvy), np.repeat(y, prob.nvx), np.outer(wy, wx).ravel()


def _mesh(prob):
    """Cells with up to four edges, counter-clockwise: per (cell, edge) the
    neighbour (-1 outside), face index, outward normal, length, midpoint minus
    centroid and boundary side; per face its first cell and edge."""
    if prob.unstructured:
        ids = np.asarray(prob.cell_nodes)
        sides = np.asarray(prob.edge_side)
        real = np.where(ids < 0, ids[:, :1], ids)
        P = np.stack([np.asarray(prob.nodes_x)[real], np.asarray(prob.nodes_y)[real]], -1)
        count = np.where(ids[:, 3] < 0, 3, 4)
    else:
        ni, nj = prob.ni, prob.nj
        j, i = (q.ravel() for q in np.meshgrid(np.arange(nj), np.arange(ni), indexing="ij"))
        ci, cj = np.stack([i, i + 1, i + 1, i], 1), np.stack([j, j, j + 1, j + 1], 1)
        P = np.stack([prob.nodes_x[cj, ci], prob.nodes_y[cj, ci]], -1)
        pi, pj = prob.bc[I.IMIN][0] == I.BC_PERIODIC, prob.bc[I.JMIN][0] == I.BC_PERIODIC
        ids = (cj % nj if pj else cj) * (ni + 1) + (ci % ni if pi else ci)
        sides = np.stack([np.where(j == 0, I.JMIN, -1), np.where(i == ni - 1, I.IMAX, -1),
                          np.where(j == nj - 1, I.JMAX, -1), np.where(i == 0, I.IMIN, -1)], 1)
        count = np.full(len(i), 4)
    N = len(P)
    O = P - P[:, :1]
    nxt = [(m + 1) % 4 for m in range(4)]
    cr = O[:, :, 0] * O[:, nxt, 1] - O[:, nxt, 0] * O[:, :, 1]  # a triangle's repeated node adds nothing
    area = 0.5 * cr.sum(1)
    cen = ((O + O[:, nxt]) * cr[..., None]).sum(1) / (6.0 * area[:, None])
    nb = np.full((N, 4), -1)
    face = np.full((N, 4), -1)
    sign = np.zeros((N, 4))
    nrm, length, r = np.zeros((N, 4, 2)), np.zeros((N, 4)), np.zeros((N, 4, 2))
    first, seen = [], {}
    for c in range(N):
        k = count[c]
        for m in range(k):
            q = (m + 1) % k
            t = P[c, q] - P[c, m]
            length[c, m] = math.sqrt(t[0] * t[0] + t[1] * t[1])
            nrm[c, m] = (t[1] / length[c, m], -t[0] / length[c, m])
            r[c, m] = 0.5 * (O[c, m] + O[c, q]) - cen[c]
            a, b = int(ids[c, m]), int(ids[c, q])
            # (a periodic direction few cells wide folds edges of both directions onto the same nodes)
            key = (min(a, b), max(a, b), 0 if prob.unstructured else m % 2)
            if key in seen:
                f = seen[key]
                c2, m2 = first[f]
                nb[c, m], nb[c2, m2], face[c, m], sign[c, m] = c2, c, f, -1.0
            else:
                seen[key] = face[c, m] = len(first)
                sign[c, m] = 1.0
                first.append((c, m))
    g = np.zeros((N, 4, 2))
    d = np.zeros((N, 4, 2))
    for c, m in zip(*np.nonzero(nb >= 0)):
        f = face[c, m]
        c1, m1 = first[f]
        if sign[c, m] > 0:  # the neighbour is the face's second cell
            c2 = nb[c, m]
            m2 = [q for q in range(4) if face[c2, q] == f and sign[c2, q] < 0][0]
            d[c, m] = r[c, m] - r[c2, m2]
        else:
            d[c, m] = r[c, m] - r[c1, m1]
    a11, a12, a22 = (d[..., 0] ** 2).sum(1), (d[..., 0] * d[..., 1]).sum(1), (d[..., 1] ** 2).sum(1)
    det = a11 * a22 - a12 * a12
    ok = det > (1e-10 * (a11 + a22) ** 2 if prob.unstructured else 0.0)
    inv = np.where(ok, 1.0 / np.where(ok, det, 1.0), 0.0)[:, None]
    g[..., 0] = (a22[:, None] * d[..., 0] - a12[:, None] * d[..., 1]) * inv
    g[..., 1] = (a11[:, None] * d[..., 1] - a12[:, None] * d[..., 0]) * inv
    return dict(N=N, area=area, nb=nb, face=face, sign=sign, n=nrm, S=length, r=r, g=g, sides=sides,
                first=np.array(first), h=area / length.max(1), cen=P[:, 0] + cen)


def _levels(nb, lower):
    N = len(nb)
    lev = np.zeros(N, dtype=int)
    for c in (range(N) if lower else range(N - 1, -1, -1)):
        for b in nb[c]:
            if b >= 0 and (b < c if lower else b > c):
                lev[c] = max(lev[c], lev[b] + 1)
    order = np.argsort(lev, kind="stable")
    return np.split(order, np.cumsum(np.bincount(lev))[:-1])


class _Scheme:
    def __init__(self, prob, mixed):
        self.p, self.mixed, self.dev = prob, mixed, _device()
        self.m = _mesh(prob)
        x, y, w = _velocities(prob)
        t = self.t = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=self.dev)
        self.x, self.y, self.w = t(x), t(y), t(w)
        xi = np.sqrt(x * x + y * y).max()
        self.dt = prob.cfl_phys * self.m["h"].min() / xi
        self.hs = 0.5 * self.dt
        self.dtimp = prob.cfl_imp * self.m["h"] / xi
        om = prob.omega
        self.mu = 15.0 * math.sqrt(2.0 * math.pi * prob.RT_ref) * prob.Kn / (2.0 * (5.0 - 2.0 * om) * (7.0 - 2.0 * om))
        self.Pr = prob.Pr if prob.shakhov else 1.0
        one, s2 = torch.ones_like(self.x), self.x ** 2 + self.y ** 2
        self.psiG = torch.stack([one, self.x, self.y, self.x ** 2, self.x * self.y, self.y ** 2, self.x * s2,
                                 self.y * s2], 1) * self.w[:, None]
        self.levels = [_levels(self.m["nb"], True), _levels(self.m["nb"], False)]
        self.nbt = torch.as_tensor(self.m["nb"], device=self.dev)
        # faces: first cell and, inside, the second
        first = self.m["first"]
        self.fL, self.mL = first[:, 0], first[:, 1]
        self.nf = len(first)
        self.fR, self.mR = np.full(self.nf, -1), np.zeros(self.nf, dtype=int)
        for c, m in zip(*np.nonzero(self.m["sign"] < 0)):
            self.fR[self.m["face"][c, m]], self.mR[self.m["face"][c, m]] = c, m
        self.side = np.where(self.fR < 0, self.m["sides"][self.fL, self.mL], -1)
        self.iters = 0
        self.wallS = None

    # state -----------------------------------------------------------------
    def uniform(self):
        rho, u, v, T = self.p.init
        RT = T * self.p.RT_ref
        one = torch.ones(self.m["N"], 1, dtype=torch.float64, device=self.dev)
        self.f = torch.stack(self.maxwell(rho * one, u * one, v * one, RT * one))
        self.W = np.tile([rho, rho * u, rho * v, 0.5 * rho * (u * u + v * v + (self.p.K + 2) * RT)], (self.m["N"], 1))

    def maxwell(self, rho, u, v, RT):
        g = rho / (2.0 * math.pi * RT) * torch.exp(-((self.x - u) ** 2 + (self.y - v) ** 2) / (2.0 * RT))
        return g, self.p.K * RT * g

    def shakhov(self, rho, u, v, RT, qx, qy):
        """Columns of per-cell numbers -> the equilibrium pair on all velocities."""
        rho, u, v, RT, qx, qy = (self.t(q)[:, None] for q in (rho, u, v, RT, qx, qy))
        g, h = self.maxwell(rho, u, v, RT)
        if self.p.shakhov:
            cx, cy = self.x - u, self.y - v
            c = (cx * qx + cy * qy) * ((1.0 - self.p.Pr) / ((self.p.K + 4) * rho * RT * RT))
            e = (cx * cx + cy * cy) / RT
            g, h = g * (1.0 + c * (e - 4.0)), h * (1.0 + c * (e - 2.0))
        return torch.stack([g, h])

    def raw(self, f):
        return torch.cat([f[0] @ self.psiG, f[1] @ self.psiG[:, :3]], 1).cpu().numpy()

    def heat(self, r, u, v):
        """1/2 int c (c^2 G + H) about (u, v)."""
        U2 = u * u + v * v
        sx = (r[:, 6] - 2 * u * r[:, 3] - 2 * v * r[:, 4] + U2 * r[:, 1] - u * (r[:, 3] + r[:, 5])
              + 2 * u * u * r[:, 1] + 2 * u * v * r[:, 2] - u * U2 * r[:, 0])
        sy = (r[:, 7] - 2 * u * r[:, 4] - 2 * v * r[:, 5] + U2 * r[:, 2] - v * (r[:, 3] + r[:, 5])
              + 2 * u * v * r[:, 1] + 2 * v * v * r[:, 2] - v * U2 * r[:, 0])
        return 0.5 * (sx + r[:, 9] - u * r[:, 8]), 0.5 * (sy + r[:, 10] - v * r[:, 8])

    def prim(self, W):
        rho, u, v = W[:, 0], W[:, 1] / W[:, 0], W[:, 2] / W[:, 0]
        return rho, u, v, (2.0 * W[:, 3] / rho - u * u - v * v) / (self.p.K + 2)

    def tau(self, rho, RT):
        return self.mu * (RT / self.p.RT_ref) ** self.p.omega / (rho * RT)

    def cell_q(self):
        rho, u, v, RT = self.prim(self.W)
        tau = self.tau(rho, RT)
        k = 2.0 * tau / (2.0 * tau + self.dt * self.Pr)
        qx, qy = self.heat(self.raw(self.f), u, v)
        return rho, u, v, RT, tau, k * qx, k * qy

    def moments(self):
        rho, u, v, RT, _, qx, qy = self.cell_q()
        return np.stack([rho, u, v, RT / self.p.RT_ref, qx, qy], 1)

    # one iteration -----------------------------------------------------------
    def slopes(self, fb):
        m, N = self.m, self.m["N"]
        g = self.t(m["g"])
        sx, sy = torch.zeros_like(fb), torch.zeros_like(fb)
        hi, lo = fb.clone(), fb.clone()
        for q in range(4):
            has = self.nbt[:, q] >= 0
            near = fb[:, torch.where(has, self.nbt[:, q], torch.arange(N, device=self.dev))]
            sx += g[:, q, 0, None] * (near - fb)
            sy += g[:, q, 1, None] * (near - fb)
            if self.p.limiter:
                hi, lo = torch.maximum(hi, near), torch.minimum(lo, near)
        if self.p.limiter:
            phi = torch.ones_like(fb)
            r = self.t(m["r"])
            for q in range(4):
                there = torch.as_tensor(m["face"][:, q] >= 0, device=self.dev)[:, None]
                inc = sx * r[:, q, 0, None] + sy * r[:, q, 1, None]
                x = torch.where(inc > 0, hi - fb, lo - fb) / torch.where(inc == 0, torch.ones_like(inc), inc)
                th = (x * x + 2.0 * x) / (x * x + x + 2.0)
                phi = torch.where((inc != 0) & there, torch.minimum(phi, th), phi)
            sx, sy = sx * phi, sy * phi
        return sx, sy

    def side_maxwell(self, sd):
        kind, rho, u, v, T = self.p.bc[sd]
        q = [torch.full((1, 1), z, dtype=torch.float64, device=self.dev) for z in
             (rho if kind == I.BC_FARFIELD else 1.0, u, v, T * self.p.RT_ref)]
        return torch.stack(self.maxwell(*q))

    def faces(self, fb, sx, sy):
        """Fluxes (f xi.n S) of every face along its first cell's normal, and their moments."""
        m = self.m
        F = torch.empty(2, self.nf, len(self.x), dtype=torch.float64, device=self.dev)
        psi = torch.stack([torch.ones_like(self.x), self.x, self.y, 0.5 * (self.x ** 2 + self.y ** 2)], 1) * self.w[:, None]
        Phi = np.zeros((self.nf, 4))
        ghost = []
        step = max(64, int(2e7) // len(self.x))
        for a in range(0, self.nf, step):
            ix = np.arange(a, min(self.nf, a + step))
            L, R, n = self.fL[ix], self.fR[ix], m["n"][self.fL[ix], self.mL[ix]]
            s = self.t(n[:, :1]) * self.x + self.t(n[:, 1:]) * self.y

            def rec(c, mm):
                rr = self.t(m["r"][c, mm])
                cc = torch.as_tensor(c, device=self.dev)
                return fb[:, cc] + sx[:, cc] * (rr[:, :1] - self.x * self.hs) + sy[:, cc] * (rr[:, 1:] - self.y * self.hs)

            left = rec(L, self.mL[ix])
            right = rec(np.maximum(R, 0), self.mR[ix])
            for sd in range(4):
                at = np.nonzero(self.side[ix] == sd)[0]
                if not len(at):
                    continue
                M = self.side_maxwell(sd)
                at_t = torch.as_tensor(at, device=self.dev)
                ss = s[at_t]
                if self.p.bc[sd][0] == I.BC_WALL:
                    out = (self.w * ss.clamp(min=0) * left[0, at_t]).sum(1)
                    inn = (self.w * (-ss).clamp(min=0) * M[0]).sum(1)
                    right[:, at_t] = M * (out / inn)[None, :, None]
                    if self.p.implicit_wall:
                        S0 = (self.w * ss.clamp(min=0) * self.f[0, torch.as_tensor(L[at], device=self.dev)]).sum(1)
                        ghost.append((ix[at], M, ss, S0, inn))
                else:
                    right[:, at_t] = M.expand(2, len(at), -1)
            fbar = torch.where(s > 0, left, torch.where(s < 0, right, 0.5 * (left + right)))
            del left, right
            r = self.raw(fbar)
            rho, u, v = r[:, 0], r[:, 1] / r[:, 0], r[:, 2] / r[:, 0]
            RT = ((r[:, 3] + r[:, 5] + r[:, 8]) / rho - u * u - v * v) / (self.p.K + 2)
            rho0, T0 = self.p.init[0], self.p.init[3]
            # mixed precision takes an unresolved (evacuated) face as free transport
            empty = ~((rho > 1e-6 * rho0) & (RT > 1e-6 * T0 * self.p.RT_ref)) if self.mixed else np.zeros(len(rho), bool)
            rho, RT = np.where(empty, rho0, rho), np.where(empty, T0 * self.p.RT_ref, RT)
            u, v = np.where(empty, 0.0, u), np.where(empty, 0.0, v)
            tau = self.tau(rho, RT)
            qx, qy = self.heat(r, u, v)
            k = 2.0 * tau / (2.0 * tau + self.hs * self.Pr)
            wa = self.t(np.where(empty, 1.0, 2.0 * tau / (2.0 * tau + self.hs)))[:, None]
            eq = self.shakhov(rho, u, v, RT, k * qx, k * qy)
            Fl = (wa * fbar + (1.0 - wa) * eq) * s * self.t(m["S"][L, self.mL[ix]])[:, None]
            F[:, a:a + len(ix)] = Fl
            ph = (Fl[0] @ psi).cpu().numpy()
            ph[:, 3] += 0.5 * (Fl[1] @ self.w).cpu().numpy()
            Phi[ix] = ph
        for q in range(self.nf):
            if self.side[q] >= 0 and self.p.bc[self.side[q]][0] == I.BC_WALL:
                Phi[q, 0] = 0.0
        # linearised wall: the last iteration's change of the wall's mass flux re-enters as a ghost increment
        if self.p.implicit_wall:
            last, self.wallS = self.wallS, {}
            for ix, M, ss, S0, inn in ghost:
                for q, z in zip(ix.tolist(), S0.tolist()):
                    self.wallS[q] = z
                if last is not None:
                    drho = (S0 - torch.tensor([last[q] for q in ix.tolist()], dtype=torch.float64, device=self.dev)) / inn
                    SS = self.t(m["S"][self.fL[ix], self.mL[ix]])[:, None]
                    F[:, torch.as_tensor(ix, device=self.dev)] += ss.clamp(max=0) * SS * drho[:, None] * M
        return F, Phi

    def predictor(self, Phi):
        m, p = self.m, self.p
        N, nb = m["N"], m["nb"]
        gam = (p.K + 4) / (p.K + 2)
        RW = -(m["sign"][..., None] * Phi[m["face"]]).sum(1)
        rho, u, v, RT = self.prim(self.W)
        cs = np.sqrt(gam * RT)
        E = np.where(nb >= 0, nb, np.arange(N)[:, None])
        un = 0.5 * (u[:, None] + u[E]) * m["n"][..., 0] + 0.5 * (v[:, None] + v[E]) * m["n"][..., 1]
        lam = (np.abs(un) + 0.5 * (cs[:, None] + cs[E])) * m["S"]
        other = nb != np.arange(N)[:, None]
        D = m["area"] / self.dtimp + 0.5 * p.lusgs_omega * (lam * other).sum(1)
        pr = (gam - 1.0) * (self.W[:, 3] - 0.5 * rho * (u * u + v * v))
        S = 0.5 * m["S"]

        def off(c, use, dW):
            """Sum over the neighbours in `use` of 1/2 (dF S - omega Lambda dW)."""
            b = E[c]
            d, n0, n1 = dW[b], m["n"][c][..., 0], m["n"][c][..., 1]
            r0, u0, v0 = rho[b], u[b], v[b]
            ir = 1.0 / (r0 + d[..., 0])
            du, dv = (d[..., 1] - u0 * d[..., 0]) * ir, (d[..., 2] - v0 * d[..., 0]) * ir
            dvn = du * n0 + dv * n1
            vn = u0 * n0 + v0 * n1 + dvn
            dp = (gam - 1.0) * (d[..., 3] - 0.5 * (d[..., 1] * (u0 + du) + d[..., 2] * (v0 + dv) + r0 * u0 * du + r0 * v0 * dv))
            dF = np.stack([d[..., 0] * vn + r0 * dvn, d[..., 1] * vn + r0 * u0 * dvn + dp * n0,
                           d[..., 2] * vn + r0 * v0 * dvn + dp * n1,
                           (d[..., 3] + dp) * vn + (self.W[b, 3] + pr[b]) * dvn], -1)
            t = S[c][..., None] * dF - 0.5 * p.lusgs_omega * lam[c][..., None] * d
            return (t * use[..., None]).sum(1)

        dW = np.zeros((N, 4))
        cells = np.arange(N)
        if p.relax_sweeps:
            use = (nb >= 0) & other
            for _ in range(p.relax_sweeps):
                dW = (RW - off(cells, use, dW)) / D[:, None]
            return RW, dW
        low, up = (nb >= 0) & (nb < cells[:, None]), nb > cells[:, None]
        for c in self.levels[0]:
            dW[c] = (RW[c] - off(c, low[c], dW)) / D[c, None]
        for c in self.levels[1]:
            dW[c] -= off(c, up[c], dW) / D[c, None]
        return RW, dW

    def sweeps(self, R, Dc):
        """Micro LU-SGS: increments from the residual R with D = Dc + the outflow."""
        m = self.m
        cells = np.arange(m["N"])[:, None]
        nx, ny = self.t(m["n"][..., 0] * m["S"]), self.t(m["n"][..., 1] * m["S"])
        other = self.t((m["nb"] != cells) * (m["face"] >= 0))
        masks = [self.t((m["nb"] >= 0) & (m["nb"] < cells)), self.t(m["nb"] > cells)]
        E = self.nbt.clamp(min=0)
        d = R
        for forward in (True, False):
            mask = masks[0 if forward else 1]
            for c in self.levels[0 if forward else 1]:
                c = torch.as_tensor(c, device=self.dev)
                a = nx[c][..., None] * self.x + ny[c][..., None] * self.y  # [n][4][Nv]
                D = Dc[c][:, None] + (a.clamp(min=0) * other[c][..., None]).sum(1)
                coef = (-a).clamp(min=0) * mask[c][..., None]
                inc = torch.stack([(coef * d[q][E[c]]).sum(1) for q in (0, 1)])
                d[:, c] = (d[:, c] + inc) / D if forward else d[:, c] + inc / D
        return d

    def cell_stage(self):
        """fb+ of Eq. (12), its slopes, fluxes."""
        rho, u, v, RT, tau, qx, qy = self.cell_q()
        eq = self.shakhov(rho, u, v, RT, qx, qy)
        c1 = self.t((2.0 * tau - self.hs) / (2.0 * tau + self.dt))[:, None]
        fb = c1 * self.f + (1.0 - c1) * eq
        F, Phi = self.faces(fb, *self.slopes(fb))
        return tau, qx, qy, eq, F, Phi

    def net(self, F):
        """Sum over a cell's faces of the outward flux."""
        face, sign = torch.as_tensor(np.maximum(self.m["face"], 0), device=self.dev), self.t(self.m["sign"])
        return sum(sign[:, q, None] * F[:, face[:, q]] for q in range(4))

    def iterate(self):
        m = self.m
        _, qx, qy, _, F, Phi = self.cell_stage()
        RW, dW = self.predictor(Phi)
        self.W = self.W + dW
        rho, u, v, RT = self.prim(self.W)
        cq = self.t(2.0 * m["area"] / (2.0 * self.tau(rho, RT) + self.dt))
        R = -self.net(F) - cq[:, None] * (self.f - self.shakhov(rho, u, v, RT, qx, qy))
        del F
        self.f = self.f + self.sweeps(R, self.t(m["area"] / self.dtimp) + cq)
        self.Phi = Phi
        return math.sqrt(((RW / m["area"][:, None]) ** 2).sum())

    def explicit(self):
        if not self.iters:
            r = self.raw(self.f)
            self.W = np.stack([r[:, 0], r[:, 1], r[:, 2], 0.5 * (r[:, 3] + r[:, 5] + r[:, 8])], 1)
        self.iters += 1
        tau, _, _, eq, F, Phi = self.cell_stage()
        b = self.t(2.0 * self.dt / (2.0 * tau + self.dt))[:, None]
        self.f = (1.0 - b) * self.f + b * eq - self.t(self.dt / self.m["area"])[:, None] * self.net(F)
        r = self.raw(self.f)
        self.W = np.stack([r[:, 0], r[:, 1], r[:, 2], 0.5 * (r[:, 3] + r[:, 5] + r[:, 8])], 1)

    # results ---------------------------------------------------------------
    def wall_faces(self, sd):
        return [(f, self.fL[f], self.mL[f]) for f in range(self.nf) if self.side[f] == sd]

    def wall(self, sd):
        rows = []
        _, _, u, v, _ = self.p.bc[sd]
        for f, c, m in self.wall_faces(sd):
            n, P = self.m["n"][c, m], self.Phi[f] / self.m["S"][c, m]
            mid = self.m["cen"][c] + self.m["r"][c, m]
            rows.append([mid[0], mid[1], P[1] * n[0] + P[2] * n[1], P[2] * n[0] - P[1] * n[1], P[3] - u * P[1] - v * P[2]])
        return np.array(rows)

    def force(self, sd):
        return sum(self.Phi[f, 1:3] for f, _, _ in self.wall_faces(sd))


def exact(case, seed):
    if case["kind"] == "adjoint":
        return None  # the transposed solve has no short independent statement
    probs = _problems(case, seed)
    mixed = case["prec"] == "mixed"
    if case["kind"] == "batch":  # the first three instances; the others would take minutes
        out = []
        for p in probs[:3]:
            s = _Scheme(p, mixed)
            s.uniform()
            for _ in range(case["iters"]):
                s.iterate()
            out.append(s.moments())
        return out + [None] * (len(probs) - 3)
    s = _Scheme(probs[0], mixed)
    s.uniform()
    if case["kind"] == "state":
        G, H, W = _start_state(probs[0], seed)
        s.f, s.W = torch.stack([G, H]), W.cpu().numpy()
    first = None
    for _ in range(case["iters"]):
        r = s.explicit() if case.get("explicit") else s.iterate()
        if case["kind"] == "solve":
            first = first or r
            if r <= case["tol"] * first:
                break
    if case["kind"] == "state":
        return {"G": s.f[0].cpu().numpy(), "H": s.f[1].cpu().numpy(), "W": s.W}
    out = {"moments": s.moments()}
    if case["prec"] == "fp64":
        out["G"], out["H"], out["W"] = s.f[0].cpu().numpy(), s.f[1].cpu().numpy(), s.W
    if case["kind"] == "solve":
        out["wall"] = s.wall(I.JMAX)
    elif case["flow"] == "cylinder":
        out["wall"], out["drag"] = s.wall(I.JMIN), s.force(I.JMIN)
    return out
