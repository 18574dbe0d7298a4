"""The solver's performance cases: what a program that uses this library has it do.

A pass advances a flow by a few time steps through the public entry points and
reads the updated fields (and, for a single handle, the energy-balance
diagnostics) back, as a program that saves or plots every few steps does:

  single   ``Solver`` + ``qslbm_step`` + ``qslbm_observables`` with fields
  batch    ``Batch.step`` + every member's state
  serve    ``Server``: submit, run until answered, poll, fields, release

Sizes: the 2-D Hartmann channel, the 64x64x128 and 96x96x512 pipes, the batched
and the served mixes of ``paper_2211_09370_gb300.workloads``, whose boxes are
(D + 8)^2 x a few D.  Every flow starts from the Ha = 0 profile with 1 % seeded
noise inside the wall (the served requests' start), so that a pass works on a
developed flow.  FP32 handles keep FP32 fields; the library hands them out
widened to binary64, and a pass narrows them back to the type they have.

``exact`` is the method written in plain torch in binary64 (single-step flow
update with GZS forcing, tau_m = 1 magnetic sweeps, explicit immersed
boundary), independent of the library.
"""
from __future__ import annotations

import ctypes as C
import math
import random

import numpy as np
import torch

from paper_2211_09370_gb300 import _lib

SINGLE = dict(kind="single", dim=3, alpha=1.0, flow_q=19, field="uniform", precision="fp32", n_mag_cap=270,
              force_amp=0.0)


def listed():
    def one(name, **kw):
        return dict(SINGLE, name=name, **kw)

    return [
        # the 2-D Hartmann channel (64x32, FP64, uncapped N_mag = 465): the smallest solve, all latency
        one("channel_64x32_fp64", dim=2, nx=64, ny=32, nz=1, D=31.0, Re=10.0, Ha=10.0, Rm=1e-2, precision="fp64",
            n_mag_cap=0, steps=4),
        # the smallest served pipe solved alone (D = 16, box 24^2 x 96)
        one("pipe16", nx=24, ny=24, nz=96, D=16.0, Re=100.0, Ha=20.0, Rm=1e-3, steps=10),
        # the next served size alone (D = 32, box 40^2 x 192): more planes than the GPU has SMs
        one("pipe32", nx=40, ny=40, nz=192, D=32.0, Re=200.0, Ha=40.0, Rm=1e-3, steps=10),
        # the benchmark pipe (64x64x128, D = 56), FP32
        one("pipe64", nx=64, ny=64, nz=128, D=56.0, Re=100.0, Ha=20.0, Rm=1e-3, steps=10),
        # the same pipe in plain FP64, the accuracy reference users compare with
        one("pipe64_fp64", nx=64, ny=64, nz=128, D=56.0, Re=100.0, Ha=20.0, Rm=1e-3, precision="fp64", steps=2),
        # an odd box from the batched range (D = 49), ramped field: nothing divides anything
        one("pipe49_odd", nx=57, ny=57, nz=245, D=49.0, Re=300.0, Ha=30.0, Rm=2e-3, field="tanh", steps=5),
        # a six-pole in-plane applied field and the D3Q27 flow lattice on the benchmark grid
        one("magnets64_q27", nx=64, ny=64, nz=128, D=56.0, Re=100.0, Ha=20.0, Rm=1e-3, field="poles", flow_q=27,
            steps=5),
        # the large ramped pipe (96x96x512, D = 88), pulsating force; fields exceed L2
        one("ramp96", nx=96, ny=96, nz=512, D=88.0, Re=500.0, Ha=50.0, Rm=1e-2, field="tanh", force_amp=0.2,
            steps=4),
        # the same at Rm = 1 (18 sweeps per step): force, flow and diagnostics weigh more
        one("ramp96_rm1", nx=96, ny=96, nz=512, D=88.0, Re=500.0, Ha=50.0, Rm=1.0, field="tanh", force_amp=0.2,
            steps=20),
        # twelve small pipes advanced together (the served mix's small sizes)
        dict(name="batch12_small", kind="batch", count=12, mix=5, dmin=16, dmax=20, lmin=4.0, lmax=6.0,
             precision="fp32", steps=8),
        # eight uneven pipes of the batched range (D in [24, 80], L in [4D, 8D])
        dict(name="batch8_uneven", kind="batch", count=8, mix=4, dmin=24, dmax=80, lmin=4.0, lmax=8.0,
             precision="fp32", steps=2),
        # requests through the server: admitted, advanced 20 steps, read and released
        dict(name="serve6", kind="serve", count=6, mix=7, dmin=16, dmax=24, lmin=4.0, lmax=6.0, precision="fp32",
             steps=20),
    ]


def _loguni(rng, a, b):
    return math.exp(rng.uniform(math.log(a), math.log(b)))


def draw(rng):
    kind = rng.choices(("single", "batch", "serve"), (7, 2, 1))[0]
    if kind == "single":
        D = float(round(_loguni(rng, 14, 96)))
        fp64 = rng.random() < 0.2
        nx, ny = int(D) + rng.randint(7, 11), int(D) + rng.randint(7, 10)
        nz = round(D * _loguni(rng, 1.5, 6.5))
        nz = max(8, min(nz, (1_000_000 if fp64 else 4_700_000) // (nx * ny)))
        Rm = _loguni(rng, 1e-4, 1.0)
        c = dict(SINGLE, nx=nx, ny=ny, nz=nz, D=D, Re=round(_loguni(rng, 50, 500), 1), Ha=round(rng.uniform(0, 60), 1),
                 Rm=Rm, precision="fp64" if fp64 else "fp32", field=rng.choice(("uniform", "uniform", "tanh", "poles")),
                 flow_q=rng.choice((19, 19, 19, 27)), alpha=rng.choice((1.0, 1.0, 0.75)),
                 force_amp=rng.choice((0.0, 0.2)))
        most = (0.5e9 if fp64 else 4.5e9) / (nx * ny * nz * _units(c)["n_mag"])
        c["steps"] = max(1, min(10, int(most)))
        return c
    lo = rng.randint(14, 40)
    if kind == "serve":
        return dict(kind="serve", count=rng.randint(2, 6), mix=rng.randrange(1 << 20), dmin=lo // 2 + 6, dmax=24,
                    lmin=2.0, lmax=6.0, precision="fp32", steps=rng.randint(10, 20))
    return dict(kind="batch", count=rng.randint(2, 9), mix=rng.randrange(1 << 20), dmin=lo, dmax=lo + rng.randint(2, 24),
                lmin=2.0, lmax=7.0, precision=rng.choice(("fp32", "fp32", "fp32", "fp64")), steps=1)


# ------------------------------------------------------------- the problems
def _members(case):
    """The members' single-handle cases of a batch or a set of requests."""
    rng = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        D = float(rng.randint(case["dmin"], case["dmax"]))
        nz = round(D * rng.uniform(case["lmin"], case["lmax"]))
        if case["precision"] == "fp64":
            nz = min(nz, round(2.5 * D))
        out.append(dict(SINGLE, nx=int(D) + 8, ny=int(D) + 8, nz=nz, D=D, Re=_loguni(rng, 30, 500),
                        Ha=rng.uniform(0, 60), Rm=_loguni(rng, 1e-4, 1e-2), field=rng.choice(("uniform", "tanh")),
                        precision=case["precision"], steps=case["steps"]))
    return out


def _poles(c):
    """In-plane applied field of six alternating poles, [3][ny][nx]: the ideal
    sextupole inside the pipe, its wall value's size outside."""
    x = np.arange(c["nx"])[None, :] - (c["nx"] - 1) / 2.0
    y = np.arange(c["ny"])[:, None] - (c["ny"] - 1) / 2.0
    s = np.maximum(x * x + y * y, (c["D"] / 2.0) ** 2)
    return np.stack([(x * x - y * y) / s, -2.0 * x * y / s, np.zeros_like(s)])


def _params(c, seed):
    p = dict(dim=c["dim"], nx=c["nx"], ny=c["ny"], nz=c["nz"], geometry="channel" if c["dim"] == 2 else "pipe",
             diameter=c["D"], Re=c["Re"], Ha=c["Ha"], Rm=c["Rm"], b0_dir=(0.0, 1.0, 0.0) if c["dim"] == 2 else (1.0, 0.0, 0.0),
             n_mag_cap=c["n_mag_cap"], precision=c["precision"], alpha=c["alpha"], seed=seed, perturb=0.01,
             init_kind="poiseuille", flow_q=c["flow_q"] if c["dim"] == 3 else 0)
    if c["field"] == "tanh":
        p.update(b0_kind="tanh", ramp_center=c["nz"] / 2.0, ramp_width=16.0)
    elif c["field"] == "poles":
        p.update(b0_kind="field", b0_field=_poles(c))
    if c["force_amp"]:
        p.update(force_amp=c["force_amp"], force_period=2000.0)
    return p


def _nodes(c):
    return c["nx"] * c["ny"] * c["nz"]


class _Fields:
    """A program's own buffers for one instance's fields: the binary64 arrays
    the library fills (page-locked) and, for an FP32 handle, their narrowed copy."""

    def __init__(self, c):
        n = _nodes(c)
        self.wide = [torch.empty((k, c["nz"], c["ny"], c["nx"]), dtype=torch.float64, pin_memory=True)
                     for k in (1, 3, 3)]
        self.ptr = [C.cast(w.data_ptr(), C.POINTER(C.c_double)) for w in self.wide]
        self.own = [torch.empty(w.shape, dtype=torch.float32) for w in self.wide] if c["precision"] == "fp32" else self.wide
        assert n == self.wide[0].numel()

    def out(self):
        if self.own is not self.wide:
            for a, w in zip(self.own, self.wide):
                a.copy_(w)
        return {"rho": self.own[0], "u": self.own[1], "b": self.own[2]}


def prepare(case, seed):
    L = _lib.load()
    if case["kind"] == "single":
        return {"case": case, "L": L, "solver": _lib.Solver(_params(case, seed)), "fields": _Fields(case),
                "obs": _lib.qslbm_obs()}
    members = _members(case)
    params = [_params(c, seed * 64 + i) for i, c in enumerate(members)]
    if case["kind"] == "batch":
        return {"case": case, "L": L, "batch": _lib.Batch(params), "fields": [_Fields(c) for c in members]}
    # a server holding a budget that fits all requests; every pass sends them anew
    return {"case": case, "params": params,
            "server": _lib.Server(hbm_budget_bytes=4 << 30, chunk_steps=case["steps"], precision=case["precision"])}


def run(state):
    case = state["case"]
    if case["kind"] == "single":
        s, f, o = state["solver"], state["fields"], state["obs"]
        s.step(case["steps"])
        _lib.check(state["L"].qslbm_observables(s.h, C.byref(o), *f.ptr), "qslbm_observables")
        return dict(f.out(), E_k=o.E_k, E_m=o.E_m, pump=o.pump, visc=o.visc, joule=o.joule, nan=int(o.nan_flag))
    if case["kind"] == "batch":
        b = state["batch"]
        b.step(case["steps"])
        for i, f in enumerate(state["fields"]):
            m = b.member(i)
            _lib.check(state["L"].qslbm_get_state(m.h, *f.ptr, None), "qslbm_get_state")
        return [f.out() for f in state["fields"]]
    srv = state["server"]
    ids = [srv.submit(p, tol=1e-12, max_steps=case["steps"], keep_fields=True) for p in state["params"]]
    left, answers = set(ids), {}
    while left:
        srv.run()
        for r in srv.poll():
            left.discard(r["id"])
            answers[r["id"]] = r["steps"]
    out = []
    for i in ids:
        rho, u, b = srv.fields(i)
        srv.release(i)
        f = {"rho": rho[None], "u": u, "b": b}
        out.append(dict({k: v.astype(np.float32) for k, v in f.items()} if case["precision"] == "fp32" else f,
                        steps=int(answers[i])))
    return out


def work(case):
    """Bytes: the state (rho, u, b) read once and written once in its own type.
    Floating-point operations per node: a sweep 51 (flux 12, neighbour sums 24,
    update 15), the force 20 and the flow update 60 per lattice direction."""
    bytes_ = flops = 0.0
    for c in ([case] if case["kind"] == "single" else _members(case)):
        q = (c["flow_q"] if c["dim"] == 3 else 9) - 1
        bytes_ += 2.0 * 7 * (8 if c["precision"] == "fp64" else 4) * _nodes(c)
        flops += float(c["steps"]) * _nodes(c) * (51.0 * _units(c)["n_mag"] + 80.0 * q)
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------ exact (binary64)
def _units(c):
    """Lattice-unit values of the problem (L = D/2)."""
    R = 0.5 * c["D"]
    U0 = min(0.05, c["Re"] / (6.0 * R), c["Re"] * R / (2.0 * c["Ha"] ** 2) if c["Ha"] > 0 else 1.0)
    nu, eta = U0 * R / c["Re"], U0 * R / c["Rm"]
    cm2 = 1.0 / 3.0 if c["dim"] == 2 else 0.25
    cmag = 2.0 * eta / cm2
    near = round(cmag)
    n = near if abs(cmag - near) <= 1e-12 * cmag else math.ceil(cmag)
    n = max(1, min(n, c["n_mag_cap"]) if c["n_mag_cap"] > 0 else n)
    return dict(R=R, U0=U0, nu=nu, eta=eta, tau=3.0 * nu + 0.5, B0=c["Ha"] * math.sqrt(eta * nu) / R, cm2=cm2,
                F0=(2.0 if c["dim"] == 2 else 4.0) * nu * U0 / (R * R), lm=eta / (0.5 * cm2), n_mag=n)


def _lattice(q):
    """(velocity, weight) of the moving directions, and the rest weight."""
    axes = (0, 1) if q == 9 else (0, 1, 2)
    w = {9: (4 / 9, 1 / 9, 1 / 36, 0), 19: (1 / 3, 1 / 18, 1 / 36, 0), 27: (8 / 27, 2 / 27, 1 / 54, 1 / 216)}[q]
    r = (-1, 0, 1)
    dirs = [(x, y, z) for x in r for y in r for z in (r if 2 in axes else (0,))]
    return [(d, w[sum(map(abs, d))]) for d in dirs if any(d) and w[sum(map(abs, d))] > 0], w[0]


def _at(f, d):
    """f at x + d (components first; z, y, x last)."""
    return torch.roll(f, (-d[2], -d[1], -d[0]), (-3, -2, -1))


class _Exact:
    def __init__(self, c, seed):
        self.c, self.un = c, _units(c)
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        nx, ny, nz, R = c["nx"], c["ny"], c["nz"], self.un["R"]
        cx, cy = (nx - 1) / 2.0, (ny - 1) / 2.0
        z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij", sparse=True)
        d2 = ((y - cy) ** 2 if c["dim"] == 2 else (x - cx) ** 2 + (y - cy) ** 2) + 0.0 * (x + z)
        self.dist = np.sqrt(d2)
        inside = self.dist <= R
        # noise: splitmix64 of seed ^ (3 k + component), the top 53 bits to [-1, 1)
        self.axis = 0 if c["dim"] == 2 else 2
        u = np.zeros((3, nz, ny, nx))
        k = np.arange(nx * ny * nz, dtype=np.uint64).reshape(nz, ny, nx)
        with np.errstate(over="ignore"):
            for a in range(c["dim"]):
                s = (np.uint64(seed) ^ (k * np.uint64(3) + np.uint64(a))) + np.uint64(0x9E3779B97F4A7C15)
                s = (s ^ (s >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
                s = (s ^ (s >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
                s = s ^ (s >> np.uint64(31))
                u[a] = np.where(inside, 0.01 * self.un["U0"] * ((s >> np.uint64(11)).astype(float) * 2.0 ** -52 - 1.0), 0)
        u[self.axis] += np.where(inside, self.un["U0"] * (1.0 - d2 / (R * R)), 0.0)
        self.u = self.t(u.astype(np.float32).astype(float) if c["precision"] == "fp32" else u)
        self.drho = torch.zeros((1, nz, ny, nx), dtype=torch.float64, device=self.dev)
        self.b = torch.zeros_like(self.u)
        if c["field"] == "tanh":
            be = np.zeros((3, nz, 1, 1))
            be[0, :, 0, 0] = 0.5 * (1.0 + np.tanh((np.arange(nz) - nz / 2.0) / 16.0))
        elif c["field"] == "poles":
            be = _poles(c)[:, None]
        else:
            be = np.zeros((3, 1, 1, 1))
            be[1 if c["dim"] == 2 else 0] = 1.0
        self.be = self.t(self.un["B0"] * be)
        self.time = 0
        self._markers(cx, cy)

    def t(self, a):
        return torch.as_tensor(a, device=self.dev)

    def _markers(self, cx, cy):
        """One plane's wall markers (every plane carries the same): 3 x 3
        supports and weights of the three-point Lagrange kernel, and the scalings."""
        c, R = self.c, self.un["R"]
        if c["dim"] == 2:
            X = np.concatenate([np.arange(c["nx"])] * 2).astype(float)
            Y = np.repeat([cy - R, cy + R], c["nx"])
        else:
            n = round(math.pi * c["D"])
            th = 2.0 * math.pi * np.arange(n) / n
            X, Y = cx + R * np.cos(th), cy + R * np.sin(th)

        def line(v):
            n0 = np.floor(v + 0.5)
            n0 = np.where(n0 - v > 0.5, n0 - 1, np.where(n0 - v <= -0.5, n0 + 1, n0))
            r = n0 - v
            return n0.astype(int), np.stack([0.5 * r * (r + 1), 1 - r * r, 0.5 * r * (r - 1)], 1)

        (ix, wx), (iy, wy) = line(X), line(Y)
        o = np.arange(-1, 2)
        q = ((iy[:, None] + o) % c["ny"])[:, :, None] * c["nx"] + ((ix[:, None] + o) % c["nx"])[:, None, :]
        w = wy[:, :, None] * wx[:, None, :]
        W = np.zeros(c["nx"] * c["ny"])
        np.add.at(W, q.ravel(), w.ravel())
        d = (w * W[q]).sum((1, 2))
        lm = self.un["lm"]
        self.q, self.w = self.t(q.reshape(-1)), self.t(w.reshape(-1, 9))
        self.su, self.sb = self.t(1.0 / d), self.t(lm / (d * (1.0 + d * (lm - 1.0))))

    def _wall(self, f, s):
        g = f.view(3, self.c["nz"], -1)
        v = g[:, :, self.q].view(3, self.c["nz"], -1, 9)
        delta = -s * (v * self.w).sum(-1)
        g.index_add_(2, self.q, (delta[..., None] * self.w).flatten(2))

    def _sweep(self, w0, w1, kappa):
        u, b = self.u, self.b
        B = self.be + b
        e = torch.stack([u[0] * B[1] - u[1] * B[0], u[0] * B[2] - u[2] * B[0], u[1] * B[2] - u[2] * B[1]])
        X, Y, Z = (1, 0, 0), (0, 1, 0), (0, 0, 1)
        neg = lambda d: tuple(-v for v in d)  # noqa: E731
        s = _at(b, X) + _at(b, neg(X)) + _at(b, Y) + _at(b, neg(Y))
        ex = _at(e[:2], neg(X)) - _at(e[:2], X)
        ey = _at(e[::2], neg(Y)) - _at(e[::2], Y)
        D = torch.stack([-ey[0], ex[0], ex[1] + ey[1]])
        if self.c["dim"] == 3:
            s += _at(b, Z) + _at(b, neg(Z))
            D[:2] += _at(e[1:], Z) - _at(e[1:], neg(Z))
        self.b = w0 * b + w1 * (s + kappa * D)

    def _curl(self, b, dirs):
        g = [torch.zeros_like(b) for _ in range(3)]
        for d, w in dirs:
            nb = _at(b, d)
            for a in range(3):
                if d[a]:
                    g[a] += 3.0 * w * d[a] * nb
        return torch.stack([g[1][2] - g[2][1], g[2][0] - g[0][2], g[0][1] - g[1][0]])

    def _body(self):
        a = self.c["force_amp"]
        return self.un["F0"] * (1.0 + a * math.sin(2.0 * math.pi * self.time / 2000.0) if a else 1.0)

    def step(self):
        c, un = self.c, self.un
        a = c["alpha"]
        w0, w1 = ((0.25, 0.125) if c["dim"] == 3 else (1 / 3, 1 / 6))
        for _ in range(un["n_mag"]):
            self._sweep((w0 - 1 + a) / a, w1 / a, 1.0 / (2.0 * un["eta"]))
            self._wall(self.b, self.sb)
        dirs, wr = _lattice(c["flow_q"] if c["dim"] == 3 else 9)
        F = torch.linalg.cross(self._curl(self.b, dirs), self.be + self.b, dim=0)
        F[self.axis] += self._body()
        u, tau = self.u, un["tau"]
        uu = (u * u).sum(0, keepdim=True)
        rho = 2.0 * wr * (self.drho - 1.5 * uu * (1 + self.drho)) - self.drho
        m = torch.zeros_like(u)
        for d, w in dirs:
            dr, un_, Fn = _at(self.drho, d), _at(u, d), _at(F, d)
            cv = torch.tensor(d, dtype=torch.float64, device=self.dev).view(3, 1, 1, 1)
            cu, cF = (cv * un_).sum(0, keepdim=True), (cv * Fn).sum(0, keepdim=True)
            sq = 4.5 * cu * cu - 1.5 * (un_ * un_).sum(0, keepdim=True)
            f = w * (dr + (1 + dr) * (3.0 * cu + sq))
            fb = w * (dr + (1 + dr) * (sq - 3.0 * cu))
            rho += 0.5 * f + 1.5 * fb
            gz = (1.0 - 0.5 / tau) * w * (18.0 * cu * cF - 6.0 * (un_ * Fn).sum(0, keepdim=True))
            m += cv * ((tau - 1.0) * f - tau * fb - 0.5 * tau * gz)
        m += F - 2.0 * (tau - 1.0) * (1.0 + self.drho) * u
        self.drho, self.u = rho, m / (1.0 + rho)
        self._wall(self.u, self.su)
        self.time += 1

    def fields(self):
        return {"rho": (1.0 + self.drho).cpu(), "u": self.u.cpu(), "b": self.b.cpu()}

    def balance(self):
        c = self.c
        mask = self.t(self.dist <= self.un["R"] - 2.0).double()
        mean = lambda f: float((f * mask).sum() / mask.sum())  # noqa: E731
        dirs, _ = _lattice(c["flow_q"] if c["dim"] == 3 else 9)
        lap = sum(w * (_at(self.u, d) - self.u) for d, w in dirs)
        B = self.be + self.b
        jxb = torch.linalg.cross(self._curl(self.b, dirs), B, dim=0)
        return {"E_k": mean(0.5 * (1 + self.drho[0]) * (self.u ** 2).sum(0)), "E_m": mean(0.5 * (B ** 2).sum(0)),
                "pump": mean(self._body() * self.u[self.axis]),
                "visc": -self.un["nu"] * mean((self.u * 6.0 * lap).sum(0)), "joule": -mean((self.u * jxb).sum(0))}


def exact(case, seed):
    def after(c, seed):
        e = _Exact(c, seed)
        for _ in range(c["steps"]):
            e.step()
        return e

    if case["kind"] == "single":
        e = after(case, seed)
        return dict(e.fields(), **e.balance(), nan=None)
    return [dict(after(c, seed * 64 + i).fields(), **({"steps": None} if case["kind"] == "serve" else {}))
            for i, c in enumerate(_members(case))]
