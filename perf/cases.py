"""Measured cases of the solver: jobs as a program that uses the library runs them.

A pass is one job through the public entry points: an initial velocity field
that is on the GPU goes into a solver (``Solver.set_state``), the solver takes
the case's steps (``Solver.step`` or ``Ensemble.step``), and the program reads
the force rows and the velocity back (``forces``, ``get_state_device``).  The
solver with its workspace is made once and kept, as a program keeps it; the
start of the job is part of the pass, so a pass on a state gives the same
outputs each time.

The initial field is a mean inflow plus random-phase, divergence-free modes
with a -5/3 spectrum, the inflow of the turbulent-insect workload, from the
seed.  ``exact`` takes the same steps in FP64 with plain torch operations: full
half spectra, ``torch.fft``, the mask formulas point by point.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1506_06513_gb300 as fl
import workloads

DEVICE = "cuda"
DEG = math.pi / 180.0

# Every case names: the grid n = nx x ny x nz, the longest side of the box
# (cubic cells), the precision, the time scheme, the steps of a job, the body,
# and whether the wake terms (vorticity sponge and Dirichlet inflow layer) are
# on.  members > 1: an ensemble of that many independent flapping wings.
_BASE = {"nx": 0, "ny": 0, "nz": 0, "box": 4.0, "precision": "fp32", "scheme": "ab2", "steps": 1,
         "body": "model", "wake": False, "members": 1, "re": 300.0}


def _case(name, n, steps, **kw):
    c = dict(_BASE, nx=n[0], ny=n[1], nz=n[2], steps=steps, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain-method check: 32^3 FP64, a fixed sphere with the tanh layer
        # in a 2 pi box, 20 steps; the smallest job, where launches and latency
        # count
        _case("sphere_32_fp64", (32, 32, 32), 20, box=2 * math.pi, precision="fp64", body="tanh_sphere"),
        # a small insect on an uneven grid (the size of the parity tests), as
        # run while a set-up is being tried out
        _case("insect_48x36x24_fp32", (48, 36, 24), 20),
        # a parameter study: 40 flapping wings of their own amplitude,
        # frequency and Reynolds number on small grids of four kinds, together
        _case("ensemble_40_fp32", (0, 0, 0), 30, body="wing", members=40),
        # one flapping wing at Re = 100, the middle size
        _case("wing_256_fp32", (256, 256, 256), 10, body="wing", re=100.0),
        # the model insect at Re = 300 in inflow: the headline workload
        _case("insect_512_fp32", (512, 512, 512), 10),
        # the same with the x transforms on the tensor cores
        _case("insect_512_bf16x2", (512, 512, 512), 5, precision="bf16x2"),
        # the largest: the insect in turbulent inflow at Re = 1000
        _case("turbulent_1024_fp32", (1024, 1024, 1024), 3, re=1000.0),
        # the reference precision at the middle size
        _case("insect_256_fp64", (256, 256, 256), 3, precision="fp64"),
        # the paper's falling-sphere grid: free flight, sponge and inflow
        # layer, lengths that are no power of two
        _case("falling_384x384x768_fp32", (384, 384, 768), 3, box=8.0, body="falling", wake=True),
        # contour wings, head and eyes under RK4, three factors of length 192
        _case("realistic_rk4_192_fp32", (192, 192, 192), 3, body="realistic", scheme="rk4"),
        # radix 3 only, odd y and z lengths and mode counts
        _case("wing_162x81x243_fp32", (162, 81, 243), 10, body="wing", re=100.0),
        # RK4 at the headline's row length with the wake terms, in a flat box
        _case("wake_rk4_512x128x96_fp32", (512, 128, 96), 2, scheme="rk4", wake=True, body="sphere"),
    ]


SMOOTH = sorted(2 ** a * 3 ** b for a in range(11) for b in range(7) if 8 <= 2 ** a * 3 ** b <= 1024)
ENSEMBLE_GRIDS = ((64, 64, 64), (96, 96, 96), (128, 128, 128), (96, 96, 192))
_COST = {"fp32": 1.0, "fp64": 20.0, "bf16x2": 1.3, "bf16x3": 1.5}


def draw(rng):
    """One more case: sizes over the logarithm of the whole range, all lengths
    2^a 3^b, the four precisions, both schemes, every body, with and without
    the wake terms; at most a third of the largest listed case's work."""
    if rng.random() < 0.15:
        return _case("", (0, 0, 0), rng.randint(5, 20), body="wing", members=rng.randint(2, 40))
    precision = rng.choice(("fp32", "fp32", "fp32", "fp64", "bf16x2", "bf16x3"))
    top = 1.0e9 / _COST[precision]              # grid points times steps
    lo, hi = math.log(12.0), math.log(min(768.0, top ** (1 / 3)))

    def near(x):
        return min(SMOOTH, key=lambda v: abs(math.log(v) - x))

    while True:
        x = rng.uniform(lo, hi)
        if precision.startswith("bf16"):
            nx = rng.choice((256, 512))
            x = min(math.log(nx), x)
        else:
            nx = near(x + rng.uniform(-0.4, 0.4))
        ny, nz = near(x + rng.uniform(-0.5, 0.5)), near(x + rng.uniform(-0.5, 0.5))
        if nx % 2 == 0 and nx * ny * nz <= top:
            break
    scheme = rng.choice(("ab2", "ab2", "rk4"))
    stages = 4 if scheme == "rk4" else 1
    most = max(1, min(20, int(top / (nx * ny * nz * stages))))
    slim = min(nx, ny, nz) * 2 < max(nx, ny, nz)     # no room for a wing span
    body = rng.choice(("sphere",) if slim else ("sphere", "wing", "model", "realistic"))
    return _case("", (nx, ny, nz), rng.randint(1, most), precision=precision, scheme=scheme, body=body,
                 wake=rng.random() < 0.3, re=round(math.exp(rng.uniform(math.log(50.0), math.log(1000.0))), 3))


# ------------------------------------------------------------------- inputs

def _members(case, seed):
    """(configuration, insect descriptor) of every run of the case."""
    out = []
    rng = np.random.default_rng([6513, seed])
    for i in range(case["members"]):
        phi, freq, re = 60.0 * DEG, 1.0, case["re"]
        n, box = (case["nx"], case["ny"], case["nz"]), case["box"]
        if case["members"] > 1:
            n = ENSEMBLE_GRIDS[i % 4]
            box = 8.0 if n[2] == 192 else 4.0
            phi, freq, re = rng.uniform(40, 80) * DEG, rng.uniform(0.8, 1.2), rng.uniform(50, 400)
        dx = box / max(n)
        L = tuple(dx * v for v in n)
        span = min(1.0, 0.45 * min(L))
        mean = (0.25, 0.0, 0.0)
        # with C_eta fixed a coarse grid would put less than a point into the
        # penalization layer; scale it with the cell as the fine grids have it
        cfg = {"name": "case", "n": n, "L": L, "nu": workloads.nu_from_re(re, 4 * phi * freq, 0.3),
               "eta": max(5e-4, 0.128 * dx), "cfl": 0.1, "mean_mode": "fixed", "u_inf": mean,
               "time_scheme": case["scheme"], "force_ring": 64}
        if case["wake"]:
            cfg.update(sponge_c=0.1, sponge_width=(8.5 * dx, 8.5 * dx, 0.0), layer_width=(4.5 * dx, 0.0, 0.0))
        centre = tuple(0.5 * v for v in L)
        body = case["body"]
        if body in ("sphere", "tanh_sphere"):
            ins = workloads.sphere(centre, (0.25 if body == "sphere" else 0.08) * min(L),
                                   profile="cos" if body == "sphere" else "tanh")
        elif body == "falling":
            ins = workloads.sphere((centre[0], centre[1], 0.75 * L[2]), 0.5, profile="cos")
            ins["free_flight"] = {"mass": 1.5, "gravity": 1.0, "J_body": (0.1, 0.1, 0.1),
                                  "dof": (1.0, 1.0, 1.0, 0.0, 0.0, 0.0)}
        elif body == "wing":
            ins = workloads.single_wing(L, n, phi_m=phi, freq=freq)
            ins["wing"] = (0.15 * span, 0.15 * span, span, 4 * dx)
        else:
            ins = workloads.realistic_insect(L, n) if body == "realistic" else workloads.model_insect(L, n)
            ins["wing"] = (0.15, 0.15, 1.0, 4 * dx)
        out.append((cfg, ins))
    return out


def _field(cfg, seed, k):
    """[3][nz][ny][nx] FP32 on the GPU: the mean plus every mode with
    2 <= |k| <= 8 (those the grid resolves), random phases, divergence free,
    -5/3 spectrum, u_rms 0.1."""
    n, L = cfg["n"], cfg["L"]
    rng = np.random.default_rng([1506, seed, k])
    top = [min(int(8.0 * L[j] / (2 * math.pi)), n[j] // 3) for j in range(3)]
    m = np.stack(np.meshgrid(*(np.arange(-t, t + 1) for t in top), indexing="ij"), -1).reshape(-1, 3)
    half = (m[:, 0] > 0) | ((m[:, 0] == 0) & ((m[:, 1] > 0) | ((m[:, 1] == 0) & (m[:, 2] > 0))))
    kv = 2 * math.pi * m / np.array(L)
    kk = np.sqrt((kv ** 2).sum(1))
    keep = half & (kk >= 2.0) & (kk <= 8.0)
    if not keep.any():                       # a box too small for that band: its first modes
        keep = half & (np.abs(m).max(1) <= 1)
    kv, kk = kv[keep], kk[keep]
    a = rng.standard_normal((len(kk), 3)) + 1j * rng.standard_normal((len(kk), 3))
    a -= kv * ((kv * a).sum(1) / kk ** 2)[:, None]
    a *= (kk ** (-5.0 / 6.0 - 1.0))[:, None]
    a *= 0.1 * math.sqrt(3.0) / math.sqrt(2 * (np.abs(a) ** 2).sum())
    ax = [np.exp(1j * np.outer(np.arange(n[j]) * (L[j] / n[j]), kv[:, j])) for j in range(3)]   # (n_j, M)
    ex, ey, ez = (torch.as_tensor(v, dtype=torch.complex64, device=DEVICE) for v in ax)
    amp = torch.as_tensor(2 * a, dtype=torch.complex64, device=DEVICE)
    u = torch.empty((3, n[2], n[1], n[0]), dtype=torch.float32, device=DEVICE)
    planes = max(1, min(n[2], (1 << 22) // (n[1] * len(kk)) + 1))
    for c in range(3):
        right = (ex * amp[:, c]).T.contiguous()                                                  # (M, nx)
        for z0 in range(0, n[2], planes):
            left = ez[z0:z0 + planes, None, :] * ey[None, :, :]
            u[c, z0:z0 + planes] = torch.matmul(left, right).real + cfg["u_inf"][c]
    return u


class _State:
    pass


def prepare(case, seed):
    st = _State()
    st.steps = case["steps"]
    st.single = case["precision"] != "fp64"
    st.sims, st.u, st.out = [], [], []
    for k, (cfg, ins) in enumerate(_members(case, seed)):
        st.sims.append(fl.Solver(cfg, ins, precision=case["precision"]))
        u = _field(cfg, seed, k)
        st.u.append(u if st.single else u.double())
        st.out.append(torch.empty_like(st.u[-1]))
    torch.cuda.synchronize()
    st.ens = None
    if len(st.sims) > 1:
        for s, u in zip(st.sims, st.u):
            s.set_state(u)                       # an ensemble is made of solvers that hold a state
        st.ens = fl.Ensemble(st.sims)
    return st


def run(st):
    for s, u in zip(st.sims, st.u):
        s.set_state(u)
    if st.ens is not None:
        st.ens.step(st.steps)
    else:
        st.sims[0].step(st.steps)
    rows = [s.forces(64)[0] for s in st.sims]
    for s, o in zip(st.sims, st.out):
        s.get_state_device(o)
    # the rows of a single-precision run carry no more than its fields do
    rows = np.stack(rows).astype(np.float32 if st.single else np.float64)
    return {"u": list(st.out), "rows": rows}


def _modes(n):
    return (n[0] // 3 + 1) * (2 * (n[1] // 3) + 1) * (2 * (n[2] // 3) + 1)


def work(case):
    """Bytes: the initial and the final field once, and per right-hand side the
    state and one more field of the scheme (the previous or the stage term)
    read and written once, kept modes only.  Flops: per right-hand side nine
    real 3-D transforms at 2.5 N log2 N and 60 operations a point."""
    size = 8 if case["precision"] == "fp64" else 4
    stages = 4 if case["scheme"] == "rk4" else 1
    byt = flop = 0.0
    for i in range(case["members"]):
        n = (case["nx"], case["ny"], case["nz"]) if case["members"] == 1 else ENSEMBLE_GRIDS[i % 4]
        N = float(n[0] * n[1] * n[2])
        byt += size * (6 * N + case["steps"] * stages * 4 * 3 * 2 * _modes(n))
        flop += (6 + 9 * case["steps"] * stages) * 2.5 * N * math.log2(N) + 60 * N * case["steps"] * stages
    return {"bytes": byt, "flops": flop}


# ------------------------------------- the same job in FP64 with plain torch

def _rot(axis, a, d=False):
    """Rotation into a frame turned by `a` about an axis, or its derivative."""
    c, s = (-math.sin(a), math.cos(a)) if d else (math.cos(a), math.sin(a))
    i, j = ((1, 2), (2, 0), (0, 1))[axis]
    m = np.zeros((3, 3))
    m[axis, axis] = 0.0 if d else 1.0
    m[i, i] = m[j, j] = c
    m[i, j], m[j, i] = s, -s
    return m


def _angle(series, f, t):
    a0, a, b = series
    v, d = 0.5 * a0, 0.0
    for i, (p, q) in enumerate(zip(a, b)):
        w = 2 * math.pi * (i + 1) * f
        v += p * math.cos(w * t) + q * math.sin(w * t)
        d += w * (q * math.cos(w * t) - p * math.sin(w * t))
    return v, d


def _wings(ins, t):
    """Per wing: (global-to-wing matrix, angular velocity, pivot); the body frame is the global one."""
    out = []
    for s in range(ins.get("nwings", 0)):
        sg = 1.0 if s == 0 else -1.0
        kin = ins["kinematics"]
        (phi, dphi), (al, dal), (th, dth) = (_angle(kin[k], ins["freq"], t) for k in ("phi", "alpha", "theta"))
        stroke = _rot(1, ins["eta_stroke"])
        if s == 1:
            stroke = _rot(0, math.pi) @ stroke
        A, T, P = _rot(1, sg * al), _rot(2, -th), _rot(0, sg * phi)
        dM = (_rot(1, sg * al, True) * (sg * dal) @ T @ P - A @ _rot(2, -th, True) * dth @ P
              + A @ T @ (_rot(0, sg * phi, True) * (sg * dphi))) @ stroke
        M = A @ T @ P @ stroke
        W = dM.T @ M                                   # the cross-product matrix of the angular velocity
        pivot = np.array(ins["x_cntr"]) + np.array(ins["pivot_l" if s == 0 else "pivot_r"])
        out.append((M, np.array([W[2, 1], W[0, 2], W[1, 0]]), pivot))
    return out


def _body_distance(ins, x):
    a, b = ins["body_axes"]
    if ins["body"] == "sphere":
        return torch.sqrt(x[0] ** 2 + x[1] ** 2 + x[2] ** 2) - a
    r, ax = torch.sqrt(x[1] ** 2 + x[2] ** 2), x[0].abs()
    inside = r - b * torch.sqrt(torch.clamp(1 - (ax / a) ** 2, min=0.0))
    d = torch.where(ax <= a, inside, torch.sqrt(r ** 2 + (ax - a) ** 2))
    balls = []
    if "head" in ins:
        balls.append(ins["head"])
    if "eyes" in ins:
        (ex, ey, ez), er = ins["eyes"]
        balls += [((ex, ey, ez), er), ((ex, -ey, ez), er)]
    for (cx, cy, cz), rad in balls:
        d = torch.minimum(d, torch.sqrt((x[0] - cx) ** 2 + (x[1] - cy) ** 2 + (x[2] - cz) ** 2) - rad)
    return d


def _wing_distance(ins, x):
    cle, cte, R, h = ins["wing"]
    dz = x[2].abs() - 0.5 * h
    if "contour" in ins:
        c = ins["contour"]
        px, py = x[0] - c["center"][0], x[1] - c["center"][1]
        th = torch.atan2(py, px)
        rad = torch.full_like(th, 0.5 * c["a0"])
        for i, (p, q) in enumerate(zip(c["a"], c["b"])):
            rad += p * torch.cos((i + 1) * th) + q * torch.sin((i + 1) * th)
        return torch.maximum(dz, torch.sqrt(px ** 2 + py ** 2) - rad)
    d = torch.maximum(x[0] - cle, -x[0] - cte)
    return torch.maximum(torch.maximum(d, dz), torch.maximum(x[1] - R, -x[1]))


def _chi(ins, d, h):
    if ins["profile"] == "tanh":
        return 0.5 * (1 - torch.tanh(d / h))
    c = 0.5 * (1 + torch.cos(math.pi * (d + h) / (2 * h)))
    return torch.where(d <= -h, torch.ones_like(d), torch.where(d >= h, torch.zeros_like(d), c))


def _cross(a, b):
    return [a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]]


class _Exact:
    """The penalized step of one run: spectra over the half space, N = û at k."""

    def __init__(self, cfg, ins, u):
        self.cfg, self.ins = cfg, dict(ins)
        self.n, self.L = cfg["n"], cfg["L"]
        self.N = self.n[0] * self.n[1] * self.n[2]
        self.d = [l / m for l, m in zip(self.L, self.n)]
        dev = u.device

        def wave(j, half):
            m = torch.arange(self.n[j] // 2 + 1) if half else torch.fft.fftfreq(self.n[j], 1.0 / self.n[j]).round()
            shape = [1, 1, 1]
            shape[2 - j] = -1
            m = m.double().to(dev).reshape(shape)
            return 2 * math.pi * m / self.L[j], (m.abs() <= self.n[j] // 3)

        (kx, ox), (ky, oy), (kz, oz) = wave(0, True), wave(1, False), wave(2, False)
        self.k, self.keep = (kx, ky, kz), ox & oy & oz
        self.k2 = kx ** 2 + ky ** 2 + kz ** 2
        self.inv_k2 = torch.where(self.k2 > 0, 1.0 / self.k2.clamp(min=1e-300), torch.zeros_like(self.k2))
        self.x = [torch.arange(self.n[j], device=dev, dtype=torch.float64) * self.d[j] for j in range(3)]
        self.free = self.ins.get("free_flight")
        self.body_u = np.zeros(3)
        self.uh = self.clean(torch.stack([torch.fft.rfftn(c.double(), norm="forward") for c in u]))
        for c in range(3):
            self.uh[c, 0, 0, 0] = cfg["u_inf"][c]
        self.hist, self.t, self.dt, self.body_f, self.integrals = None, 0.0, 0.0, None, None

    def clean(self, v):
        """The 2/3 rule and the projection; the mean is held (no forcing of k = 0)."""
        v *= self.keep
        dot = (self.k[0] * v[0] + self.k[1] * v[1] + self.k[2] * v[2]) * self.inv_k2
        for c in range(3):
            v[c] -= self.k[c] * dot
        v[:, 0, 0, 0] = 0
        return v

    def back(self, vh):
        return torch.fft.irfftn(vh, s=(self.n[2], self.n[1], self.n[0]), norm="forward")

    def slab(self, j, w):
        """Grid points of axis j in the end slab of thickness w."""
        i = torch.arange(self.n[j], device=self.x[0].device, dtype=torch.float64) * (self.L[j] / self.n[j])
        return (i >= self.L[j] - w) if w > 0 else torch.zeros(self.n[j], dtype=torch.bool, device=i.device)

    def rhs(self, uh, t):
        """Projected nonlinear term, penalization and wake terms, and the sums."""
        cfg, ins = self.cfg, self.ins
        u = [self.back(uh[c]) for c in range(3)]
        w = [self.back(1j * (self.k[a] * uh[b] - self.k[b] * uh[a])) for a, b in ((1, 2), (2, 0), (0, 1))]
        h = ins.get("c_smth", 1.0) * max(self.d)
        wings = _wings(ins, t)
        centre = np.array(ins["x_cntr"])
        sums = np.zeros((3, 4, 3))
        energy = umax = 0.0
        sponge = cfg.get("sponge_c", 0.0)
        width, layer = cfg.get("sponge_width", (0, 0, 0)), cfg.get("layer_width", (0, 0, 0))
        sp, la = ([self.slab(j, v[j]) for j in range(3)] for v in (width, layer))
        step = max(1, (1 << 23) // (self.n[0] * self.n[1]))
        for z0 in range(0, self.n[2], step):
            z = slice(z0, min(z0 + step, self.n[2]))
            X = [self.x[0][None, None, :], self.x[1][None, :, None], self.x[2][z][:, None, None]]
            uu, ww = [f[z] for f in u], [f[z] for f in w]
            nl = _cross(uu, ww)
            sq = uu[0] ** 2 + uu[1] ** 2 + uu[2] ** 2
            energy += float(sq.sum())
            umax = max(umax, float(sq.max()))
            best = torch.zeros_like(uu[0])
            colour = torch.zeros_like(uu[0], dtype=torch.int8)
            us = [torch.zeros_like(uu[0]) for _ in range(3)]
            e = [X[i] - centre[i] for i in range(3)]
            parts = []
            if ins["body"] != "none":
                full = [v.expand_as(best) for v in e]
                parts.append((1, _chi(ins, _body_distance(ins, full), h), [float(v) for v in self.body_u]))
            for s, (M, om, pv) in enumerate(wings):
                r = [X[i] - pv[i] for i in range(3)]
                loc = [M[i, 0] * r[0] + M[i, 1] * r[1] + M[i, 2] * r[2] for i in range(3)]
                parts.append((2 + s, _chi(ins, _wing_distance(ins, loc), h), _cross([float(v) for v in om], r)))
            for col, chi, vel in parts:
                more = chi > best
                best = torch.where(more, chi, best)
                colour[more] = col
                for i in range(3):
                    us[i] = torch.where(more, torch.as_tensor(vel[i], dtype=best.dtype, device=best.device), us[i])
            pen = [best * (uu[i] - us[i]) for i in range(3)]
            cus = [best * us[i] for i in range(3)]
            for col, _, _ in parts:
                ref = centre if col == 1 else wings[col - 2][2]
                here = (colour == col).double()
                r = [X[i] - ref[i] for i in range(3)]
                for q, v in enumerate((pen, _cross(r, pen), cus, _cross(r, cus))):
                    sums[col - 1, q] += [float((here * v[i]).sum()) for i in range(3)]
            inlet = (la[0][None, None, :] | la[1][None, :, None] | la[2][z][:, None, None]).double() / cfg["eta"]
            for i in range(3):
                # over the velocity, which nothing reads after this
                uu[i].copy_(nl[i] - pen[i] / cfg["eta"] - inlet * (uu[i] - cfg["u_inf"][i]))
            if sponge > 0:
                inside = (sp[0][None, None, :] | sp[1][None, :, None] | sp[2][z][:, None, None]).double()
                for f in ww:
                    f.mul_(inside)
        N = torch.stack([torch.fft.rfftn(f, norm="forward") for f in u])
        del u
        if sponge > 0:
            v = torch.stack([torch.fft.rfftn(f, norm="forward") for f in w])
            for c, (a, b) in enumerate(((1, 2), (2, 0), (0, 1))):
                N[c] -= 1j * (self.k[a] * v[b] - self.k[b] * v[a]) * self.inv_k2 / sponge
        return self.clean(N), sums, energy, math.sqrt(umax), wings

    def step(self):
        cfg = self.cfg
        N, sums, energy, umax, wings = self.rhs(self.uh, self.t)
        dt = min(cfg["eta"], cfg["cfl"] * min(self.d) / umax)
        first = self.hist is None
        if cfg["time_scheme"] == "rk4":
            top = sum((2 * math.pi * (m // 3) / l) ** 2 for m, l in zip(self.n, self.L))
            dt = min(dt, 2.5 / (cfg["nu"] * top))
            visc = cfg["nu"] * self.k2
            k = N - visc * self.uh
            total = k.clone()
            for frac, weight in ((0.5, 2.0), (0.5, 2.0), (1.0, 1.0)):
                stage = self.uh + frac * dt * k
                k = self.rhs(stage, self.t + frac * dt)[0] - visc * stage
                total += weight * k
            self.uh = self.uh + dt / 6.0 * total
            self.hist = N
        else:
            r = 0.0 if first else dt / self.dt
            e1 = torch.exp(-cfg["nu"] * self.k2 * dt)
            new = e1 * (self.uh + dt * (1 + 0.5 * r) * N)
            if not first:
                new -= dt * 0.5 * r * torch.exp(-cfg["nu"] * self.k2 * (dt + self.dt)) * self.hist
            self.uh, self.hist = new, N
        dV = self.d[0] * self.d[1] * self.d[2]
        force, moment = sums[:, 0] * dV / cfg["eta"], sums[:, 1] * dV / cfg["eta"]
        ints = sums[:, 2:4] * dV
        if not first:
            force = force + (ints[:, 0] - self.integrals[:, 0]) / self.dt
            moment = moment + (ints[:, 1] - self.integrals[:, 1]) / self.dt
        row = np.zeros(26)
        row[0], row[1] = self.t, dt
        for p in range(3):
            row[2 + 6 * p:5 + 6 * p], row[5 + 6 * p:8 + 6 * p] = force[p], moment[p]
        row[20], row[21] = 0.5 * energy * dV, umax
        for s, (_, om, _) in enumerate(wings):
            row[22 + s] = -float(moment[1 + s] @ om)
        if self.free:
            # translation only (the sphere's rotations are held): AB2 with the fluid's weights
            f = np.concatenate([self.body_u, force.sum(0) / self.free["mass"]])
            f[5] -= self.free["gravity"]
            rate = f if first else (1 + 0.5 * dt / self.dt) * f - 0.5 * dt / self.dt * self.body_f
            y = np.concatenate([np.array(self.ins["x_cntr"]), self.body_u]) + dt * rate
            self.ins["x_cntr"], self.body_u, self.body_f = tuple(y[:3]), y[3:], f
        self.integrals, self.dt = ints, dt
        self.t += dt
        return row


def exact(case, seed):
    if case["nx"] * case["ny"] * case["nz"] > 1.4e8:
        return None                                  # the 1024^3 job would take longer than it is worth
    us, rows = [], []
    for k, (cfg, ins) in enumerate(_members(case, seed)):
        sim = _Exact(cfg, ins, _field(cfg, seed, k))
        rows.append([sim.step() for _ in range(case["steps"])])
        us.append(torch.stack([sim.back(sim.uh[c]) for c in range(3)]))
        del sim
    return {"u": us, "rows": np.array(rows)}
