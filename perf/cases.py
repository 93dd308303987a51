"""The work that users of this solver have it do, as timed cases.

A forward case installs a state on the device, advances it some steps and
reads the new state back (``Solver.set_state``, ``step``, ``get_state``): what
a program does that drives the solver from its own arrays or restarts a run.
A backward case is the checkpointed adjoint of such a run
(``Solver.adjoint``).  Flows, sizes and options are those of the package's
workloads, tests and benchmark: flow past a cylinder and a sphere, a freely
rotating ellipse, closed containers and periodic boxes; FP32 and FP64; upwind
and limited fluxes; explicit and semi-implicit time schemes; the BGK and
Shakhov models; direct and conservative equilibria.

The exact values come from a dense torch evaluation of the scheme in 64 bits
(geometry in numpy), written from the method's formulas without the package.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1503_04544_gb300 import dvm
from paper_1503_04544_gb300 import workloads as W

_DEV = "cuda"

# ------------------------------------------------------------------ the cases

# Keys: flow; nx, ny (nz): cells; nvx, nvy (nvz): velocities; bits: state
# precision; muscl: limited fluxes; imex, shakhov, conservative: options;
# steps of a pass; every: checkpoint spacing of the adjoint (0: forward).


def _case(flow, n, nv, bits=32, muscl=True, steps=10, every=0, name=None, **opt):
    c = dict(flow=flow, nx=n[0], ny=n[1], nz=n[2] if len(n) > 2 else 1,
             nvx=nv[0], nvy=nv[1], nvz=nv[2] if len(nv) > 2 else 1,
             bits=bits, muscl=muscl, steps=steps, every=every,
             imex=False, shakhov=False, conservative=False)
    c.update(opt)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem of the package: a periodic box in FP64, where
        # launches and host calls count as much as the kernels
        _case("bump", (32, 32), (16, 16), bits=64, muscl=False, steps=20, name="bump_fp64"),
        # a small closed container stepped many times: latency of a step with
        # cut cells
        _case("disk", (64, 64), (20, 20), steps=100, name="disk_small"),
        # the flagship: Mach-2 cylinder, limited fluxes, FP32
        _case("cylinder", (256, 256), (32, 32), steps=20, name="cylinder"),
        # the same in FP64, the reference precision of the method
        _case("cylinder", (256, 256), (32, 32), bits=64, steps=4, name="cylinder_fp64"),
        # the Shakhov model (right Prandtl number) on the same flow
        _case("cylinder", (256, 256), (32, 32), steps=10, shakhov=True, name="cylinder_shakhov"),
        # small Knudsen numbers: the semi-implicit scheme
        _case("cylinder", (256, 256), (32, 32), steps=10, imex=True, name="cylinder_imex"),
        # a coarse velocity grid with the conservative equilibrium on a
        # ragged grid, velocities not a multiple of the vector width
        _case("cylinder", (301, 187), (22, 18), steps=20, conservative=True, name="cylinder_conservative_ragged"),
        # moving obstacle: geometry rebuilt every step, upwind, larger than L2
        _case("ellipse", (512, 512), (40, 40), muscl=False, steps=10, name="ellipse"),
        # 3D: the sphere at the benchmark's velocity grid
        _case("sphere", (64, 64, 64), (20, 20, 20), steps=4, name="sphere"),
        # 3D on a ragged grid with the Shakhov model
        _case("sphere", (45, 50, 37), (14, 15, 13), steps=6, shakhov=True, name="sphere_shakhov_ragged"),
        # 3D in FP64
        _case("sphere", (40, 40, 40), (12, 12, 12), bits=64, steps=3, name="sphere_fp64"),
        # backward: gradient of a functional of the final state and the drag
        _case("cylinder", (256, 256), (32, 32), steps=20, every=10, name="adjoint"),
    ]


def _pairs(c):
    return c["nx"] * c["ny"] * c["nz"] * c["nvx"] * c["nvy"] * c["nvz"]


def draw(rng):
    log = lambda a, b: int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))  # noqa: E731
    flow = rng.choice(["bump", "disk", "box", "cylinder", "cylinder", "cylinder", "ellipse", "sphere", "sphere"])
    every = rng.choice([4, 10]) if flow == "cylinder" and rng.random() < 0.25 else 0
    bits = 64 if rng.random() < 0.3 else 32
    if flow == "sphere":
        n = [log(24, 64) for _ in range(3)]
        nv = [rng.randint(8, 20) for _ in range(3)]
    else:
        lo = 32 if flow == "bump" else 64
        n = [log(lo, 512)]
        n.append(log(max(lo, n[0] / 2), min(512, 2 * n[0])))
        nv = [rng.randint(10, 40), rng.randint(10, 40)]
    c = _case(flow, n, nv, bits=bits, muscl=rng.random() < 0.7, every=every)
    if not every:
        opt = rng.choice(["", "", "imex", "shakhov", "conservative"])
        if opt:
            c[opt] = True
    # state sizes and steps up to the largest listed ones' cost
    most = 3e7 if bits == 64 else 1e9
    while _pairs(c) > most:
        k = max((k for k in ("nx", "ny", "nz")), key=lambda k: c[k])
        c[k] = c[k] * 3 // 4
    room = (2e8 if bits == 64 else 2.5e9) / _pairs(c) / (4 if every else 1)
    c["steps"] = max(2, min(log(4, 30), int(room)))
    return c


# ------------------------------------------------------------------ the problems

def _problem(c, seed):
    """The problem dict of a case; the seed moves the obstacle a little."""
    n, rng = c["nx"], np.random.default_rng([int(seed), 1])
    flow = c["flow"]
    if flow == "bump":
        cfg = W.periodic_bump(32, 16)
    elif flow == "disk":
        cfg = W.disk_container(64, 20)
    elif flow == "box":
        cfg = W.box_container(64, 20)
    elif flow == "cylinder":
        cfg = W.cylinder_adjoint(64, 16, nseg=64, seed=int(seed)) if c["every"] else W.cylinder_mach2(64, 16)
    elif flow == "ellipse":
        cfg = W.rotating_ellipse(64, 16)
    else:
        cfg = W.sphere_mach15(24, 8)
    cfg.update({k: c[k] for k in ("nx", "ny", "nz", "nvx", "nvy", "nvz")})
    cfg.update(scheme=int(c["muscl"]), time_scheme=int(c["imex"]), model=int(c["shakhov"]),
               conservative=int(c["conservative"]))
    if c["shakhov"]:
        cfg["Pr"] = 2.0 / 3.0
    if c["imex"]:
        cfg["Kn"] = 0.005
    if flow in ("cylinder", "ellipse", "sphere"):
        for k in ("cx", "cy") + (("cz",) if cfg["dim"] == 3 else ()):
            cfg[k] += float(rng.uniform(-0.02, 0.02))
    if flow == "ellipse":
        cfg["theta"], cfg["omega"] = float(rng.uniform(0, 3)), float(rng.uniform(-1, 1))
    # Maxwellian sides of the case's size
    sides = [cfg["ny"] * cfg["nz"]] * 2 + [n * cfg["nz"]] * 2 + [n * cfg["ny"]] * 2
    for s in range(6):
        if cfg["bc"][s] == 1:
            st = np.tile(np.asarray(cfg["bc_state"][s])[:1], (sides[s], 1))
            if flow == "ellipse":
                st[:, 1] = 0.5 * (2.0 * (np.arange(cfg["ny"]) + 0.5) / cfg["ny"] - 1.0)
            cfg["bc_state"][s] = st
    return cfg


def _fields(c, cfg, seed):
    """Smooth random macroscopic fields about the free stream, per cell."""
    rng = np.random.default_rng([int(seed), 2])
    ax = [(np.arange(cfg[k]) + 0.5) / cfg[k] for k in ("nx", "ny", "nz")]
    X, Y, Z = np.meshgrid(*ax, indexing="ij")
    X, Y, Z = (a.transpose(2, 1, 0).ravel() for a in (X, Y, Z))

    def wave(amp):
        s = 0.0
        for _ in range(4):
            k = rng.integers(0, 4, 3) * [1, 1, int(cfg["dim"] == 3)]
            s = s + rng.uniform(0.4, 1.0) * np.sin(2 * np.pi * (k[0] * X + k[1] * Y + k[2] * Z) + rng.uniform(0, 6.28))
        return amp / 4 * s + 0 * X

    u = 0.0
    if c["flow"] in ("cylinder", "sphere"):
        u = float(np.asarray(cfg["bc_state"][0])[0, 1])
    elif c["flow"] == "ellipse":
        u = 0.5 * (2.0 * Y - 1.0)
    return dict(rho=1 + wave(0.3), ux=u + wave(0.3), uy=wave(0.3), uz=wave(0.3 if cfg["dim"] == 3 else 0.0),
                T=1 + wave(0.2))


def _axes(cfg):
    ks = ("x", "y", "z")[: cfg["dim"]]
    return [cfg[f"v{k}min"] + torch.arange(cfg[f"nv{k}"], dtype=torch.float64, device=_DEV)
            * ((cfg[f"v{k}max"] - cfg[f"v{k}min"]) / cfg[f"nv{k}"]) for k in ks]


def _state(c, cfg, seed):
    """Initial state in the public layout [cell][component][velocity]."""
    m = {k: torch.as_tensor(v, dtype=torch.float64, device=_DEV) for k, v in _fields(c, cfg, seed).items()}
    dt = torch.float32 if c["bits"] == 32 else torch.float64
    e = [torch.exp(-(v[None] - m[k][:, None]) ** 2 / (2 * m["T"][:, None])) / (2 * math.pi * m["T"][:, None]) ** 0.5
         for v, k in zip(_axes(cfg), ("ux", "uy", "uz"))]
    e[0] = e[0] * m["rho"][:, None]
    e = [a.to(dt) for a in e]
    nc, nv = len(m["T"]), c["nvx"] * c["nvy"] * c["nvz"]
    if cfg["dim"] == 3:
        yz = (e[2][:, :, None] * e[1][:, None, :]).reshape(nc, -1)
        return (yz[:, :, None] * e[0][:, None, :]).reshape(-1)
    F = torch.empty((nc, 2, nv), dtype=dt, device=_DEV)
    F[:, 0] = (e[1][:, :, None] * e[0][:, None, :]).reshape(nc, nv)
    # g a little off its equilibrium T/2 f
    F[:, 1] = F[:, 0] * (m["T"] / 2 * (1 + 0.1 * (m["rho"] - 1)))[:, None].to(dt)
    return F.reshape(-1)


class _Prepared:
    pass


def prepare(case, seed):
    cfg = _problem(case, seed)
    st = _Prepared()
    st.case, st.cfg = case, cfg
    st.solver = dvm.Solver(cfg, dvm.FP32 if case["bits"] == 32 else dvm.FP64)
    st.F0 = _state(case, cfg, seed)
    if case["every"]:
        g = torch.Generator(device=_DEV).manual_seed(int(seed) + 7)
        st.seed = torch.rand(st.F0.numel(), generator=g, device=_DEV, dtype=torch.float32).to(st.F0.dtype) - 0.5
        # keep the forward run's tape on the device, as long runs' users do
        st.solver.set_adjoint_tape(40 << 30)
    else:
        st.out = torch.empty_like(st.F0)
    torch.cuda.synchronize()
    return st


def run(st):
    c, s = st.case, st.solver
    if st.cfg["movable"]:
        s.set_body(st.cfg)        # a pass starts from the body's initial angle
    s.set_state(st.F0)
    if c["every"]:
        r = s.adjoint(c["steps"], c["every"], with_drag=True, seed=st.seed)
        # wall-temperature gradients in the precision of the parameters
        return dict(lambda0=r["lambda0"], gTw=r["gTw"].astype(s.dtype))
    s.step(c["steps"])
    return s.get_state(st.out)


def work(case):
    """Each step reads the state at t^n and writes it at t^{n+1}: a step needs
    the velocity sums of the whole previous one, so a state larger than the
    caches passes through memory once per step; a smaller one is read and
    written once.  A transposed step reads the state and the sensitivity and
    writes the sensitivity.  Operations per pair and component: flux
    differences (3 per axis, 9 limited) and the update; per pair the
    equilibrium and the moments."""
    dim = 3 if case["nz"] > 1 else 2
    comp = 3 - dim + 1
    pairs = float(_pairs(case))
    state = pairs * comp * case["bits"] / 8
    n = case["steps"]
    per = comp * (dim * (9 if case["muscl"] else 3) + 3) + 8 + 2 * (dim + 2)
    if case["every"]:
        return {"bytes": 5 * n * state, "flops": 3 * n * per * pairs}
    return {"bytes": 2 * state * (n if 2 * state > 120e6 else 1), "flops": n * per * pairs}


# ------------------------------------------------------------------ exact values

def _edge(p0, p1, h):
    o = h * (p0 / np.where(p0 == p1, 1.0, p0 - p1))
    return np.where((p0 > 0) & (p1 > 0), h, np.where((p0 < 0) & (p1 < 0), 0.0, np.where(p0 > 0, o, h - o)))


def _polygon(p00, p10, p11, p01, h1, h2):
    """Gas area of rectangles with nodal level-set values, and their wall edge
    (length, normal, midpoint) where the level set changes sign."""
    lo, hi = np.minimum(np.minimum(p00, p10), np.minimum(p11, p01)), np.maximum(np.maximum(p00, p10), np.maximum(p11, p01))
    cut = (lo <= 0) & (hi >= 0)
    lum, lup = _edge(p00, p01, h2), _edge(p10, p11, h2)
    lwm, lwp = _edge(p00, p10, h1), _edge(p01, p11, h1)
    frac = lambda a, b: a / np.where(a == b, 1.0, a - b)  # noqa: E731
    z = np.zeros_like(p00)
    # crossings on the edges u-, u+, w-, w+
    has = [(p00 > 0) != (p01 > 0), (p10 > 0) != (p11 > 0), (p00 > 0) != (p10 > 0), (p01 > 0) != (p11 > 0)]
    pos = [(z, h2 * frac(p00, p01)), (z + h1, h2 * frac(p10, p11)), (h1 * frac(p00, p10), z), (h1 * frac(p01, p11), z + h2)]
    assert int(np.where(cut, sum(h.astype(int) for h in has), 2).max()) == 2, "saddle cell"
    first = [np.select(has, [p[d] for p in pos], 0.0) for d in (0, 1)]
    last = [np.select(has[::-1], [p[d] for p in pos[::-1]], 0.0) for d in (0, 1)]
    eu, ew = last[0] - first[0], last[1] - first[1]
    lw = np.sqrt(eu * eu + ew * ew)
    ru, rw = 0.5 * (first[0] + last[0]), 0.5 * (first[1] + last[1])
    safe = np.where(lw > 0, lw, 1.0)
    nu, nw = (lum - lup) / safe, (lwm - lwp) / safe
    area = np.where(lo > 0, h1 * h2, np.where(cut, 0.5 * (lup * h1 + lwp * h2 + lw * (ru * nu + rw * nw)), 0.0))
    return area, np.where(cut, lw, 0.0), nu, nw, ru, rw


def _level_set(cfg, ct, st, X):
    d = [x - cfg[k] for x, k in zip(X, ("cx", "cy", "cz"))]
    s = cfg["shape"]
    if s in (1, 3, 4):
        r = np.sqrt(d[0] * d[0] + d[1] * d[1] + (d[2] * d[2] if len(d) > 2 else 0.0))
        return cfg["ra"] - r if s == 4 else r - cfg["ra"]
    if s == 2:
        xr, yr = ct * d[0] + st * d[1], -st * d[0] + ct * d[1]
        a2, b2 = cfg["ra"] ** 2, cfg["rb"] ** 2
        g, gx, gy = xr * xr / a2 + yr * yr / b2 - 1.0, 2 * xr / a2, 2 * yr / b2
        n = np.sqrt(gx * gx + gy * gy)
        return np.where(n > 0, g / np.where(n > 0, n, 1.0), -min(cfg["ra"], cfg["rb"]))
    if s == 5:
        x0, x1, y0, y1 = cfg["cx"] - cfg["ra"], cfg["cx"] + cfg["ra"], cfg["cy"] - cfg["rb"], cfg["cy"] + cfg["rb"]
        return np.minimum(np.minimum(X[0] - x0, x1 - X[0]), np.minimum(X[1] - y0, y1 - X[1]))
    return np.ones_like(X[0])


def _geometry(cfg, ct=1.0, st=0.0):
    """Cut-cell geometry: arrays in grid order (z, y, x) or (y, x)."""
    D = cfg["dim"]
    ks = ("x", "y", "z")[:D]
    n = [cfg["n" + k] for k in ks]
    h = [(cfg[k + "max"] - cfg[k + "min"]) / m for k, m in zip(ks, n)]
    nodes = [cfg[k + "min"] + np.arange(m + 1) * hh for k, m, hh in zip(ks, n, h)]
    X = [a.transpose(*range(D)[::-1]) for a in np.meshgrid(*nodes, indexing="ij")]
    phi = _level_set(cfg, ct, st, X)
    eps = 1e-10 * h[0]
    phi = np.where(phi >= 0, np.maximum(phi, eps), -np.maximum(-phi, eps))
    at = lambda *o: phi[tuple(slice(a, phi.shape[i] - 1 + a) for i, a in enumerate(o[::-1]))]  # noqa: E731
    g = dict(h=h)
    if D == 2:
        p = [at(0, 0), at(1, 0), at(1, 1), at(0, 1)]
        g["vol"], g["sw"], nx, ny, rx, ry = _polygon(*p, h[0], h[1])
        g["faces"] = [_edge(phi[:-1], phi[1:], h[1]), _edge(phi[:, :-1], phi[:, 1:], h[0])]
        g["n"], r = [nx, ny], [rx, ry]
        mean = 0.25 * (((p[0] + p[1]) + p[2]) + p[3])
    else:
        face = lambda a, b, c, d, h1, h2: _polygon(a, b, c, d, h1, h2)[0]  # noqa: E731
        P = phi
        ax = face(P[:-1, :-1], P[:-1, 1:], P[1:, 1:], P[1:, :-1], h[1], h[2])
        ay = face(P[:-1, :, :-1], P[:-1, :, 1:], P[1:, :, 1:], P[1:, :, :-1], h[0], h[2])
        az = face(P[:, :-1, :-1], P[:, :-1, 1:], P[:, 1:, 1:], P[:, 1:, :-1], h[0], h[1])
        g["faces"] = [ax, ay, az]
        w = [ax[:, :, :-1] - ax[:, :, 1:], ay[:, :-1] - ay[:, 1:], az[:-1] - az[1:]]
        sw = np.sqrt(w[0] * w[0] + w[1] * w[1] + w[2] * w[2])
        off = [(0, 0, 0), (1, 0, 0), (1, 1, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1), (1, 1, 1), (0, 1, 1)]
        p = [at(*o) for o in off]
        cnt, r = 0, [0.0, 0.0, 0.0]
        for a, b in ((0, 1), (3, 2), (4, 5), (7, 6), (0, 3), (1, 2), (4, 7), (5, 6), (0, 4), (1, 5), (3, 7), (2, 6)):
            x = (p[a] > 0) != (p[b] > 0)
            t = p[a] / np.where(p[a] == p[b], 1.0, p[a] - p[b])
            cnt = cnt + x
            for d in range(3):
                r[d] = r[d] + np.where(x, h[d] * (off[a][d] + t * (off[b][d] - off[a][d])), 0.0)
        r = [q / np.maximum(cnt, 1) for q in r]
        safe = np.where(sw > 0, sw, 1.0)
        g["n"] = [q / safe for q in w]
        mean = p[0]
        for q in p[1:]:
            mean = mean + q
        mean = 0.125 * mean
    lo, hi = np.minimum.reduce(p), np.maximum.reduce(p)
    g["type"] = np.where(lo > 0, 0, np.where(hi < 0, 2, 1))
    cut = g["type"] == 1
    if D == 3:
        g["sw"] = np.where(cut, sw, 0.0)
        vol = (ax[:, :, 1:] * h[0] + ay[:, 1:] * h[1] + az[1:] * h[2]
               + sw * (r[0] * g["n"][0] + r[1] * g["n"][1] + r[2] * g["n"][2])) / 3.0
        g["vol"] = np.where(g["type"] == 0, h[0] * h[1] * h[2], np.where(cut, vol, 0.0))
    low = [a[tuple(slice(0, -1) for _ in range(D))] for a in X]
    g["r"] = [a + b for a, b in zip(low, r)]
    g["cgas"] = mean > 0
    return g


def _masters(gn, gp):
    """(member, master) pairs of the cells that are not their own master."""
    live = (gn["type"] != 2) | (gp["type"] != 2)
    out = []
    shape = gn["type"].shape
    D = len(shape)
    for idx in np.argwhere(live & ~gn["cgas"]):
        q = tuple(idx)
        for _ in range(9):
            if gn["cgas"][q]:
                break
            F = (gn if gn["type"][q] != 2 else gp)["faces"]
            best = []
            for d in range(D):
                up = tuple(v + (1 if i == D - 1 - d else 0) for i, v in enumerate(q))
                best += [(F[d][up], d, 1), (F[d][q], d, -1)]
            m = max(b[0] for b in best)
            _, d, s = next(b for b in best if b[0] == m)
            q = tuple(v + (s if i == D - 1 - d else 0) for i, v in enumerate(q))
        out.append((np.ravel_multi_index(tuple(idx), shape), np.ravel_multi_index(q, shape)))
    return np.array(out, dtype=np.int64).reshape(-1, 2)


class _Exact:
    """The scheme in 64 bits on a dense grid; rows are (component, velocity)."""

    def __init__(self, cfg):
        self.cfg, self.D = cfg, cfg["dim"]
        self.ncomp = 2 if self.D == 2 else 1
        v = _axes(cfg)
        self.dv = 1.0
        for k in ("x", "y", "z")[: self.D]:
            self.dv *= (cfg[f"v{k}max"] - cfg[f"v{k}min"]) / cfg[f"nv{k}"]
        g = torch.meshgrid(*v[::-1], indexing="ij")[::-1]
        self.v = [a.reshape(-1) for a in g]                       # per velocity
        self.nv = len(self.v[0])
        ks = ("x", "y", "z")[: self.D]
        self.h = [(cfg[k + "max"] - cfg[k + "min"]) / cfg["n" + k] for k in ks]
        self.dt = cfg["cfl"] / sum(float(a.abs().max()) / hh for a, hh in zip(v, self.h))
        self.tau0 = math.sqrt(math.pi) / 2 * cfg["Kn"] * cfg["Lref"] / math.sqrt(2.0)
        self.theta, self.omega = cfg["theta"], cfg["omega"]
        self.moving = bool(cfg["movable"])
        self.shape = tuple(cfg["n" + k] for k in ks[::-1])
        self.nc = int(np.prod(self.shape))
        self.gn = _geometry(cfg, math.cos(self.theta), math.sin(self.theta))
        self.gp = self.gn
        self.pairs = None

    def maxwell(self, rho, u, T, rows):
        """Equilibrium (columns: cells) of component 0 at velocities `rows`."""
        c2 = sum((self.v[d][rows][:, None] - u[d][None]) ** 2 for d in range(self.D))
        return rho / (2 * math.pi * T) ** (self.D / 2) * torch.exp(-c2 / (2 * T)), c2

    def sums(self, F):
        """rho, u, T of every column of F [rows][cells]."""
        f = F[: self.nv]
        s0 = f.sum(0)
        s = [self.v[d] @ f for d in range(self.D)]
        E = (0.5 * sum(a * a for a in self.v)) @ f
        if self.ncomp == 2:
            E = E + F[self.nv:].sum(0)
        rho = s0 * self.dv
        ok = rho > 0
        safe = torch.where(ok, s0, torch.ones_like(s0))
        u = [a / safe for a in s]
        T = (2 * E / safe - sum(a * a for a in u)) / 3
        return rho, u, torch.where(ok, T, torch.ones_like(T)), ok

    def heat(self, F, u):
        q = [torch.zeros_like(u[0]) for _ in u]
        for b in range(0, self.nv, 128):
            r = slice(b, min(b + 128, self.nv))
            c = [self.v[d][r][:, None] - u[d][None] for d in range(self.D)]
            w = 0.5 * sum(a * a for a in c) * F[r]
            if self.ncomp == 2:
                w = w + F[self.nv + b: self.nv + r.stop]
            for d in range(self.D):
                q[d] += (c[d] * w).sum(0)
        return [a * self.dv for a in q]

    def conservative(self, F, rho, u, T):
        """Newton on the discrete moments of the equilibrium, cells in blocks."""
        D, n = self.D, self.D + 2
        phi = [torch.ones_like(self.v[0]), *self.v, 0.5 * sum(a * a for a in self.v)]
        phi = torch.stack(phi)                                   # [n][nv]
        out = [rho.clone(), *[a.clone() for a in u], T.clone()]
        for b in range(0, self.nc, 16384):
            k = slice(b, b + 16384)
            th = torch.stack([out[0][k], *[a[k] for a in out[1:-1]], out[-1][k]])
            tgt = phi @ F[: self.nv, k] * self.dv
            if self.ncomp == 2:
                tgt[-1] += F[self.nv:, k].sum(0) * self.dv
            for _ in range(8):
                M, c2 = self.maxwell(th[0], list(th[1:-1]), th[-1], slice(None))
                M = M * self.dv
                dM = [M / th[0]] + [M * (self.v[d][:, None] - th[1 + d]) / th[-1] for d in range(D)]
                dM.append(M * (c2 / (2 * th[-1] ** 2) - D / (2 * th[-1])))
                res, J = tgt - phi @ M, torch.stack([phi @ a for a in dM], 1)   # [n][n][cells]
                if D == 2:
                    res[-1] -= th[-1] / 2 * M.sum(0)
                    J[-1] += th[-1] / 2 * torch.stack([a.sum(0) for a in dM])
                    J[-1, -1] += 0.5 * M.sum(0)
                th = th + torch.linalg.solve(J.permute(2, 0, 1), res.T).T
            for i in range(n):
                out[i][k] = th[i]
        return out[0], out[1:-1], out[-1]

    def equilibrium(self, rho, u, T, q, rows):
        """Equilibrium of velocities `rows` for every component."""
        M, c2 = self.maxwell(rho, u, T, rows)
        if q is None:
            return [M, T / 2 * M][: self.ncomp]
        k = (1 - self.cfg["Pr"]) * sum((self.v[d][rows][:, None] - u[d][None]) * q[d] for d in range(self.D)) \
            / (5 * rho * T * T)
        if self.D == 3:
            return [M * (1 + k * (c2 / T - 5))]
        return [M * (1 + k * (c2 / T - 4)), T / 2 * M * (1 + k * (c2 / T - 2))]

    def divergence(self, F, comp, rows, gas, faces):
        """Sum of the face fluxes of every cell for velocities `rows`."""
        cfg, G = self.cfg, F.reshape(-1, *self.shape)
        total = torch.zeros_like(G)
        for d in range(self.D):
            ax = self.D - d                                      # axis of G
            n = G.shape[ax]
            v = self.v[d][rows].reshape(-1, *[1] * self.D)
            ends = []
            for s in (2 * d, 2 * d + 1):
                kind = cfg["bc"][s]
                if kind == 0:
                    ends.append(G.narrow(ax, n - 2 if s % 2 == 0 else 0, 2))
                elif kind == 2:
                    e = G.narrow(ax, 0 if s % 2 == 0 else n - 1, 1)
                    ends.append(torch.cat([e, e], ax))
                else:
                    st = torch.as_tensor(np.asarray(cfg["bc_state"][s]), device=_DEV)
                    M, _ = self.maxwell(st[:, 0], [st[:, 1 + i] for i in range(self.D)], st[:, 4], rows)
                    if comp:
                        M = st[:, 4] / 2 * M
                    side = [m for i, m in enumerate(self.shape) if i != ax - 1]
                    e = M.reshape(-1, *side).unsqueeze(ax)
                    ends.append(torch.cat([e, e], ax))
            P = torch.cat([ends[0], G, ends[1]], ax)
            AA, A, B, BB = (P.narrow(ax, o, n + 1) for o in range(4))
            pos = v > 0
            fr = torch.where(pos, A, B)
            if cfg["scheme"]:
                gp = gas
                if cfg["bc"][2 * d] == 0:
                    gp = torch.cat([gas.narrow(ax - 1, n - 2, 2), gas, gas.narrow(ax - 1, 0, 2)], ax - 1)
                else:
                    one = torch.ones_like(gas.narrow(ax - 1, 0, 1))
                    gp = torch.cat([one, one, gas, one, one], ax - 1)
                ok = gp.narrow(ax - 1, 0, n + 1) & gp.narrow(ax - 1, 1, n + 1) & gp.narrow(ax - 1, 2, n + 1) \
                    & gp.narrow(ax - 1, 3, n + 1)
                a, b = B - A, torch.where(pos, A - AA, BB - B)
                mm = torch.where(a * b > 0, torch.where(a.abs() < b.abs(), a, b), 0.0)
                w = 0.5 * (1 - v.abs() * self.dt / self.h[d]) * torch.sign(v)
                fr = fr + w * mm * ok
            fl = torch.as_tensor(faces[d], device=_DEV) * (v * fr)
            total += fl.narrow(ax, 1, n) - fl.narrow(ax, 0, n)
        return total.reshape(total.shape[0], -1)

    def step(self, F):
        cfg, nv, dev = self.cfg, self.nv, F.device
        body = cfg["shape"] != 0
        theta1 = self.theta + self.dt * self.omega if self.moving else self.theta
        if self.moving:
            self.gp = _geometry(cfg, math.cos(theta1), math.sin(theta1))
        gn, gp = self.gn, self.gp
        if self.pairs is None or self.moving:
            self.pairs = _masters(gn, gp) if body else np.zeros((0, 2), np.int64)
        k, m = (torch.as_tensor(a, device=dev) for a in self.pairs.T)
        vn, vp = (torch.as_tensor(g["vol"].ravel(), device=dev) for g in (gn, gp))
        own = torch.ones(self.nc, dtype=torch.bool, device=dev)
        own[k] = False
        own &= torch.as_tensor(((gn["type"] != 2) | (gp["type"] != 2)).ravel(), device=dev)
        Sn, Sp = (torch.where(own, a, 0.0).index_add(0, m, a[k]) for a in (vn, vp))
        if len(k):                                               # fusion
            um = m.unique()
            slot = torch.zeros(self.nc, dtype=torch.int64, device=dev)
            slot[um] = torch.arange(len(um), device=dev)
            acc = F[:, um] * vn[um]
            acc.index_add_(1, slot[m], F[:, k] * vn[k])
            acc /= Sn[um]
            F[:, um] = acc
            F[:, k] = acc[:, slot[m]]
        rho_d, u, T, ok = self.sums(F)
        live = own & ok
        imex = bool(cfg["time_scheme"])
        rho, q = rho_d, None
        one = lambda a, x=1.0: torch.where(live, a, torch.full_like(a, x))  # noqa: E731
        rho_s, T_s = one(rho), one(T)
        u_s = [one(a, 0.0) for a in u]
        if not imex:
            if cfg["model"]:
                q = [one(a, 0.0) for a in self.heat(F, u_s)]
            if cfg["conservative"]:
                Fs = F
                rho_s, u_s, T_s = self.conservative(torch.where(live, Fs, self.maxwell_rows(one)), rho_s, u_s, T_s)
        wall = None
        if body:                                                 # wall density, stress, torque
            wc = np.flatnonzero((gn["type"].ravel() == 1) & (gn["sw"].ravel() > 0))
            W_ = torch.as_tensor(wc, device=dev)
            n = [torch.as_tensor(a.ravel()[wc], device=dev) for a in gn["n"]]
            r = [torch.as_tensor(a.ravel()[wc], device=dev) - cfg[c] for a, c in zip(gn["r"], ("cx", "cy", "cz"))]
            sw = torch.as_tensor(gn["sw"].ravel()[wc], device=dev)
            uw = [-r[1] * self.omega, r[0] * self.omega] + ([torch.zeros_like(sw)] if self.D == 3 else [])
            Tw = torch.full_like(sw, cfg["Tw"])
            M1, _ = self.maxwell(torch.ones_like(sw), uw, Tw, slice(None))
            c = [self.v[d][:, None] - uw[d] for d in range(self.D)]
            cn = sum(a * b for a, b in zip(c, n))
            fw = F[:nv, W_]
            wphi = -(cn.clamp(min=0) * fw).sum(0) / (cn.clamp(max=0) * M1).sum(0)
            if self.moving:
                fv = torch.where(cn < 0, wphi * M1, torch.where(cn > 0, fw, 0.0)) * self.dv
                t = [sum((c[a] * c[b] * fv).sum(0) * n[b] for b in range(2)) * sw for a in range(2)]
                torque = float((r[0] * t[1] - r[1] * t[0]).sum())
            wall = (W_, cn, sw, wphi * M1, Tw)
        gas = torch.as_tensor(gn["type"] == 0, device=dev)
        solid_p = torch.as_tensor((gp["type"] == 2).ravel(), device=dev)
        a = torch.where(live, Sn / torch.where(Sp > 0, Sp, 1.0), 0.0)
        b = torch.where(live, self.dt / torch.where(Sp > 0, Sp, 1.0), 0.0)
        rel = 0.0 if imex else self.dt / self.tau0 * rho_d
        new = torch.empty_like(F)
        skip = torch.as_tensor((gn["type"] == 2).ravel(), device=dev)
        chunk = max(1, int(3e8 // self.nc))
        for r0 in range(0, nv, chunk):
            rows = slice(r0, min(r0 + chunk, nv))
            eq = None if imex else self.equilibrium(rho_s, u_s, T_s, q, rows)
            for comp in range(self.ncomp):
                f = F[comp * nv + r0: comp * nv + rows.stop]
                R = self.divergence(f, comp, rows, gas, gn["faces"])
                R[:, skip] = 0.0
                if wall is not None:
                    W_, cn, sw, fw, Tw = wall
                    w = fw[rows] * (Tw / 2 if comp else 1.0)
                    R[:, W_] += sw * (cn[rows].clamp(max=0) * w + cn[rows].clamp(min=0) * f[:, W_])
                if len(k):
                    R.index_add_(1, m, R[:, k])
                o = a * f - b * R
                if not imex:
                    o += a * rel * (eq[comp] - f)
                new[comp * nv + r0: comp * nv + rows.stop] = torch.where(live, o, 0.0)
        if imex:
            rho, u, T, _ = self.sums(new)
            rho, T, u = one(rho), one(T), [one(x, 0.0) for x in u]
            nu = self.dt * rho / self.tau0
            if cfg["model"]:
                q = [x / (1 + nu * cfg["Pr"]) for x in self.heat(new, u)]
            re, ue, Te = (rho, u, T)
            if cfg["conservative"]:
                re, ue, Te = self.conservative(torch.where(live, new, self.maxwell_rows(one)), rho, u, T)
            for r0 in range(0, nv, chunk):
                rows = slice(r0, min(r0 + chunk, nv))
                eq = self.equilibrium(re, ue, Te, q, rows)
                for comp in range(self.ncomp):
                    s = slice(comp * nv + r0, comp * nv + rows.stop)
                    new[s] = torch.where(live, (new[s] + nu * eq[comp]) / (1 + nu), 0.0)
        if len(k):
            new[:, k] = new[:, m]
        new[:, solid_p] = 0.0
        if self.moving:
            self.omega = self.omega + self.dt * torque / cfg["inertia"]
            self.theta, self.gn = theta1, gp
        return new

    def maxwell_rows(self, one):
        """A unit Maxwellian for columns that hold no gas."""
        z = torch.zeros(1, dtype=torch.float64, device=_DEV)
        M, _ = self.maxwell(z + 1, [z] * self.D, z + 1, slice(None))
        return torch.cat([M, M / 2][: self.ncomp])


def exact(case, seed):
    """The final state in 64 bits.  None for the adjoint: where a limiter's
    arguments are within rounding of one another its derivative depends on the
    rounding of the forward run, so the limited scheme's gradient has no value
    that another arithmetic reproduces."""
    if case["every"]:
        return None
    cfg = _problem(case, seed)
    x = _Exact(cfg)
    F = _state(case, cfg, seed).reshape(x.nc, x.ncomp * x.nv).T.to(torch.float64).contiguous()
    F[:, torch.as_tensor((x.gn["type"] == 2).ravel(), device=_DEV)] = 0.0
    for _ in range(case["steps"]):
        F = x.step(F)
    return F.T.contiguous().reshape(-1)
