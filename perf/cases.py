"""The work that users of the engine have it do, as cases that can be timed.

A case is one pass of a user's program through the public entry points: advance
an engine (or a batch of engines) by ``steps`` and read its fields back, a
whole job with upload and download, or a gradient of the inverse-wetting
problem.  Fields come back in the type that the case's storage keeps (FP64,
FP32, FP16, BF16), as a program keeps its snapshots.

``exact`` restates the method in plain torch FP64 on whole arrays
(Semprebon, Krueger, Kusumaatmaja, arXiv:1511.02155) without any of this
repository's code.
"""
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

import paper_1511_02155_gb300 as tl
from paper_1511_02155_gb300 import inverse

F64 = torch.float64
KEEP = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}


# ------------------------------------------------------------------- cases

def listed():
    return [
        # the validation run a new user starts with: a small FP64 lens, where
        # launches and the latency of one plane are everything
        dict(name="lens_64_fp64", kind="lens", nx=64, ny=64, nz=1, precision="fp64", steps=100),
        # the liquid-lens benchmark (Neumann angles), a 2-D lattice that fits in L2
        dict(name="lens_512_fp32", kind="lens", nx=512, ny=256, nz=1, precision="fp32", steps=200),
        # double emulsion on an odd lattice in half storage
        dict(name="emulsion_517_fp16", kind="emulsion", nx=517, ny=391, nz=1, precision="fp16", steps=200),
        # a whole job in a shear flow, upload to download with density and
        # velocity, at an odd size: its set-up and read-back count too
        dict(name="shear_job_1000_fp32", kind="job", nx=1000, ny=701, nz=1, precision="fp32", steps=100),
        # 2-D spinodal decomposition at a size that lives in HBM
        dict(name="spinodal_4096_fp32", kind="spinodal", nx=4096, ny=4096, nz=1, precision="fp32", steps=50),
        # walls, wells and wetting on one large 2-D lattice
        dict(name="wells_4096_fp32", kind="wells", nx=4096, ny=2048, nz=1, precision="fp32", steps=50),
        # contact-angle sweep: uneven square wells stepped as one batch
        dict(name="sweep_24_fp32", kind="sweep", count=24, nmax=768, precision="fp32", steps=100),
        # the headline 3-D quench
        dict(name="spinodal_256_fp32", kind="spinodal", nx=256, ny=256, nz=256, precision="fp32", steps=50),
        # a 3-D quench in half storage on a lattice of odd extents
        dict(name="spinodal_240_fp16", kind="spinodal", nx=240, ny=201, nz=187, precision="fp16", steps=50),
        # a 3-D drop on a wetting wall
        dict(name="drop_144_fp32", kind="drop", nx=144, ny=128, nz=80, precision="fp32", steps=50),
        # the body-force coupling in 3-D
        dict(name="forcing_128_fp32", kind="forcing", nx=128, ny=128, nz=128, precision="fp32", steps=50),
        # inverse wetting: loss and gradients through the differentiable wrapper
        dict(name="inverse_256_fp64", kind="inverse", nx=256, ny=128, nz=1, precision="fp64", steps=50, every=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lens", "emulsion", "job", "spinodal", "spinodal", "spinodal3", "spinodal3", "wells", "sweep",
                       "drop", "drop", "forcing", "forcing3", "inverse"])
    two_d = dict(nz=1, precision=rng.choice(["fp32", "fp32", "fp16", "bf16"]), steps=rng.choice([50, 100, 200]))
    if kind in ("lens", "emulsion"):
        nx = _log(rng, 48, 800)
        ny = max(40, int(nx * rng.uniform(0.4, 1.0)))
        case = dict(two_d, kind=kind, nx=nx, ny=ny)
        if nx * ny < 20000:
            case["precision"] = rng.choice(["fp64", "fp32"])
        return case
    if kind == "job":
        return dict(two_d, kind=kind, nx=_log(rng, 200, 2000), ny=_log(rng, 100, 1000), precision="fp32")
    if kind == "spinodal":
        return dict(two_d, kind=kind, nx=_log(rng, 128, 4096), ny=_log(rng, 128, 4096), steps=50)
    if kind == "spinodal3":
        n = [_log(rng, 40, 240) for _ in range(3)]
        if rng.random() < 0.5:  # 3-D users like multiples of 32 along x
            n[0] = max(64, n[0] // 32 * 32)
        return dict(kind="spinodal", nx=n[0], ny=n[1], nz=n[2], precision=rng.choice(["fp32", "fp32", "fp16", "bf16"]),
                    steps=rng.choice([20, 50]))
    if kind == "wells":
        nx = _log(rng, 512, 4096)
        return dict(two_d, kind=kind, nx=nx, ny=_log(rng, 200, 2048), precision=rng.choice(["fp32", "fp32", "fp16"]),
                    steps=50)
    if kind == "sweep":
        return dict(kind=kind, count=rng.randint(4, 32), nmax=rng.choice([256, 512, 768]), precision="fp32",
                    steps=rng.choice([50, 100]))
    if kind == "drop":
        return dict(kind=kind, nx=_log(rng, 40, 160), ny=_log(rng, 40, 160), nz=_log(rng, 24, 96),
                    precision=rng.choice(["fp32", "fp32", "bf16"]), steps=rng.choice([20, 50]))
    if kind == "forcing":
        return dict(two_d, kind=kind, nx=_log(rng, 100, 2048), ny=_log(rng, 100, 2048), precision="fp32", steps=50)
    if kind == "forcing3":
        return dict(kind="forcing", nx=_log(rng, 40, 160), ny=_log(rng, 40, 160), nz=_log(rng, 40, 160),
                    precision=rng.choice(["fp32", "fp16"]), steps=rng.choice([20, 50]))
    return dict(kind="inverse", nx=_log(rng, 64, 320), ny=_log(rng, 40, 160), nz=1, precision="fp64",
                steps=rng.randint(20, 60), every=rng.randint(5, 40))


# ------------------------------------------------------------------ inputs

def _profile(d):
    """Flat-interface profile of width alpha = 1."""
    return 0.5 * (1.0 + torch.tanh(0.5 * d))


def _grid(case):
    dev = "cuda"
    return torch.meshgrid(torch.arange(case["nz"], device=dev, dtype=F64), torch.arange(case["ny"], device=dev, dtype=F64),
                          torch.arange(case["nx"], device=dev, dtype=F64), indexing="ij")


def _uniform(seed, *shape, lo=0.0, hi=1.0):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return lo + (hi - lo) * torch.rand(*shape, generator=gen, device="cuda", dtype=F64)


def _problem(case, seed):
    """Parameters, initial fields [nz][ny][nx] on the GPU and solid mask of one engine."""
    kind, nx, ny, nz = case["kind"], case["nx"], case["ny"], case["nz"]
    r = np.random.default_rng(seed)
    p = dict(lattice=9 if nz == 1 else 19, nx=nx, ny=ny, nz=nz, alpha=1.0, tau_f=1.0, M_phi=0.1, M_psi=0.1,
             h=(0.0, 0.0, 0.0), kappa=tuple(float(v) for v in r.uniform(0.01, 0.04, 3)), coupling="pressure_tensor")
    solid, u = None, None
    if kind in ("spinodal", "forcing"):
        p.update(kappa=(0.01, 0.01, 0.01), tau_f=0.8)
        C = [1.0 / 3.0 + _uniform(3 * seed + m, nz, ny, nx, lo=-0.01, hi=0.01) for m in range(3)]
        total = C[0] + C[1] + C[2]
        C = [c / total for c in C]
        if kind == "forcing":
            p["coupling"] = "forcing"
    elif kind == "lens":
        z, y, x = _grid(case)
        R = ny / 5 * r.uniform(0.8, 1.1)
        band = 0.5 * (torch.tanh(0.5 * (y - ny / 4)) - torch.tanh(0.5 * (y - 3 * ny / 4)))
        drop = _profile(R - torch.hypot(x - nx * r.uniform(0.4, 0.6), y - 3 * ny / 4))
        C = [(1 - drop) * band, (1 - drop) * (1 - band), drop]
    elif kind in ("emulsion", "job"):
        z, y, x = _grid(case)
        d = torch.hypot(x - nx * r.uniform(0.45, 0.55), y - ny * r.uniform(0.45, 0.55))
        s = min(nx, ny) * r.uniform(0.9, 1.1)
        core, shell = _profile(0.12 * s - d), _profile(0.25 * s - d)
        C = [core, 1 - shell, shell - core]
        if kind == "job":
            u = torch.zeros(3, nz, ny, nx, device="cuda", dtype=F64)
            u[0] = 0.04 * torch.sin(2 * math.pi * y / ny)
            u[1] = 0.02 * torch.sin(2 * math.pi * x / nx)
    elif kind == "wells":
        p.update(kappa=(0.01, 0.01, 0.01), h=(0.0004, -0.0004, 0.0002))
        z, y, x = _grid(case)
        floor, block = 8, 40
        solid = (y < floor + block) | (y >= ny - 1)
        filled = torch.zeros_like(x, dtype=torch.bool)
        pitch = 128
        for k in range(nx // pitch):
            w, depth = int(r.integers(20, 80)), int(r.integers(10, 40))
            x0 = k * pitch + (pitch - w) // 2
            hole = (x >= x0) & (x < x0 + w) & (y >= floor + block - depth) & (y < floor + block)
            filled = filled | hole
        solid = solid & ~filled
        drop = torch.where(filled, _profile(floor + block - 0.5 - y), torch.zeros_like(x))
        lower = _profile(floor + block + (ny - 1 - floor - block) / 2 - y)
        C = [(1 - drop) * lower, (1 - drop) * (1 - lower), drop]
    else:  # "drop", "inverse": a fluid-3 cap on the bottom wall in fluid 1, fluid 2 under the lid
        kap = p["kappa"]
        p.update(h=tuple(float(v * k) for v, k in zip(r.uniform(-0.04, 0.04, 3), kap)), M_phi=0.3, M_psi=0.2)
        z, y, x = _grid(case)
        up, n_up = (y, ny) if nz == 1 else (z, nz)
        solid = (up < 1) | (up >= n_up - 1)
        side = (x - nx / 2) ** 2 + (0.0 if nz == 1 else (y - ny / 2) ** 2)
        R = 0.3 * min(nx, 1.5 * n_up, nx if nz == 1 else ny) * r.uniform(0.9, 1.1)
        drop = _profile(R - torch.sqrt(side + (up - 0.5) ** 2))
        lower = _profile(0.75 * n_up - up)
        C = [(1 - drop) * lower, (1 - drop) * (1 - lower), drop]
    if solid is not None:
        C = [torch.where(solid, torch.zeros_like(c), c) for c in C]
    fields = [C[0] + C[1] + C[2], C[0] - C[1], C[2]]
    return p, fields, u, solid


def _width(k, nmax):
    return 128 + 32 * int(np.random.default_rng([7, k]).integers(0, (nmax - 128) // 32 + 1))


def _well(k, seed, nmax):
    """Member k of a contact-angle sweep: a square well, half filled with fluid 3,
    and drawn wetting parameters, on a lattice whose size k alone decides."""
    nx = _width(k, nmax)
    r = np.random.default_rng([seed, k])
    case = dict(nx=nx, ny=nx // 2, nz=1)
    z, y, x = _grid(case)
    floor, width = 8, min(int(r.integers(20, 121)), nx - 16)
    top = min(floor + int(r.integers(10, 61)), case["ny"] - 4)
    x0 = (nx - width) // 2
    well = (x >= x0) & (x < x0 + width) & (y >= floor) & (y < top)
    solid = ((y < top) & ~well) | (y >= case["ny"] - 1)
    drop = torch.where(well, _profile(floor - 0.5 + 0.5 * (top - floor) - y), torch.zeros_like(x))
    lower = _profile(top + (case["ny"] - 1 - top) / 2 - y)
    C = [torch.where(solid, torch.zeros_like(x), c) for c in ((1 - drop) * lower, (1 - drop) * (1 - lower), drop)]
    h = r.uniform(-0.0012, 0.0012, 3)
    p = dict(lattice=9, nx=nx, ny=case["ny"], nz=1, kappa=(0.01, 0.01, 0.01), alpha=1.0, tau_f=1.0, M_phi=0.5,
             M_psi=1.0 / 6.0, h=tuple(float(v) for v in h - h.mean()), coupling="pressure_tensor")
    return p, [C[0] + C[1] + C[2], C[0] - C[1], C[2]], None, solid


def _host(t):
    return t.reshape(-1).cpu().numpy()


def _engine(p, precision, solid):
    eng = tl.TernaryLB(p["lattice"], p["nx"], p["ny"], p["nz"], p["kappa"], p["alpha"], p["tau_f"], p["M_phi"], p["M_psi"],
                       p["h"], None if solid is None else _host(solid), precision)
    if p["coupling"] != "pressure_tensor":
        eng.set_coupling(p["coupling"])
    return eng


def _buffers(n, keep):
    """What a program that watches its run keeps: pinned buffers for the read-back
    and the snapshot's arrays."""
    return [torch.empty(n, dtype=F64, pin_memory=True) for _ in range(3)], [torch.zeros(n, dtype=keep) for _ in range(3)]


def prepare(case, seed):
    state = dict(case=case, keep=KEEP[case["precision"]])
    if case["kind"] == "sweep":
        engines = []
        for k in range(case["count"]):
            p, fields, _, solid = _well(k, seed, case["nmax"])
            eng = _engine(p, case["precision"], solid)
            eng.init_fields(*[_host(f) for f in fields])
            engines.append(eng)
        batch = tl.TernaryBatch(engines)
        batch.set_graph(True)
        return dict(state, engines=engines, batch=batch, out=[_buffers(e.N, state["keep"]) for e in engines])
    p, fields, u, solid = _problem(case, seed)
    host = [_host(f) for f in fields]
    if case["kind"] == "inverse":
        target = fields[2] + torch.where(solid, torch.zeros_like(fields[2]), _uniform(seed + 77, *fields[2].shape, lo=-0.03, hi=0.03))
        leaves = [torch.tensor(p["kappa"], dtype=F64), torch.tensor(p["h"], dtype=F64)] + [torch.from_numpy(a.copy()) for a in host]
        return dict(state, p=p, leaves=leaves, solid=_host(solid), target=torch.from_numpy(_host(target)))
    eng = _engine(p, case["precision"], solid)
    if case["kind"] == "job":
        return dict(state, engine=eng, fields=host, u=[_host(u[a]) for a in range(3)])
    eng.init_fields(*host)
    return dict(state, engine=eng, out=_buffers(eng.N, state["keep"]))


# -------------------------------------------------------------------- pass

def _concentrations(eng, out):
    pinned, snapshot = out
    eng.fields_into(*[t.data_ptr() for t in pinned])
    for a, b in zip(snapshot, pinned):
        a.copy_(b)
    return snapshot


def run(state):
    case, keep = state["case"], state["keep"]
    if case["kind"] == "sweep":
        state["batch"].step(case["steps"])
        each = [_concentrations(e, o) for e, o in zip(state["engines"], state["out"])]
        return {"C%d" % (m + 1): torch.cat([c[m] for c in each]) for m in range(3)}
    if case["kind"] == "inverse":
        p = state["p"]
        leaves = [t.clone().requires_grad_(True) for t in state["leaves"]]
        loss = inverse.c3_misfit(*leaves, state["target"], lattice=p["lattice"], nx=p["nx"], ny=p["ny"], nz=p["nz"],
                                 alpha=p["alpha"], tau_f=p["tau_f"], M_phi=p["M_phi"], M_psi=p["M_psi"], solid=state["solid"],
                                 nsteps=case["steps"], checkpoint_every=case["every"], precision=case["precision"])
        loss.backward()
        return {"loss": loss.detach(), **{n: t.grad for n, t in zip(("kappa", "h", "rho", "phi", "psi"), leaves)}}
    eng = state["engine"]
    if case["kind"] == "job":
        eng.init_fields(*state["fields"], u=state["u"])
        eng.step(case["steps"])
        f = eng.fields()
        return {n: torch.from_numpy(a).to(keep) for n, a in f.items()}
    eng.step(case["steps"])
    out = _concentrations(eng, state["out"])
    return {"C%d" % (m + 1): out[m] for m in range(3)}


def _sizes(case):
    if case["kind"] != "sweep":
        return case["nx"] * case["ny"] * case["nz"]
    widths = [_width(k, case["nmax"]) for k in range(case["count"])]
    return sum(w * (w // 2) for w in widths)


def work(case):
    n, two_d = _sizes(case), case.get("nz", 1) == 1
    q, b = (9 if two_d else 19), BYTES[case["precision"]]
    step = 2 * 3 * q * b + (1 if case["kind"] in ("wells", "sweep", "drop", "inverse") else 0)
    flops = 450 if two_d else 1000
    if case["kind"] == "inverse":
        # forward (twice: checkpoints) and back: states read and written, the multipliers read and written
        return {"bytes": n * case["steps"] * (2 * step + 3 * 3 * q * b) + n * 8 * 7, "flops": n * case["steps"] * 5 * flops}
    read_back = 3 * q * b + 3 * 8
    if case["kind"] == "job":
        read_back = 3 * q * b * 2 + 8 * (6 + 7)  # fields in, populations out and in, fields out
    return {"bytes": n * (case["steps"] * step + read_back), "flops": n * case["steps"] * flops * (2 if case["kind"] == "forcing" else 1)}


# ---------------------------------------------------- the method in plain FP64

E9 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (1, 1, 0), (-1, -1, 0), (-1, 1, 0), (1, -1, 0)]
E19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)] + \
      [(a, b, 0) for a in (1, -1) for b in (1, -1)] + [(0, a, b) for a in (1, -1) for b in (1, -1)] + \
      [(a, 0, b) for a in (1, -1) for b in (1, -1)]


class _Exact:
    def __init__(self, p, solid, kappa=None, h=None):
        self.dim = 2 if p["lattice"] == 9 else 3
        self.E = E9 if self.dim == 2 else E19
        self.opp = [self.E.index(tuple(-c for c in e)) for e in self.E]
        w_axis, w_diag = (1 / 9, 1 / 36) if self.dim == 2 else (1 / 18, 1 / 36)
        self.W = [(4 / 9 if self.dim == 2 else 1 / 3, w_axis, w_diag)[sum(map(abs, e))] for e in self.E]
        self.solid = solid
        self.guo = p["coupling"] != "pressure_tensor"
        k = torch.tensor(p["kappa"], dtype=F64, device="cuda") if kappa is None else kappa
        hh = torch.tensor(p["h"], dtype=F64, device="cuda") if h is None else h
        self.k, self.a2 = k, p["alpha"] ** 2
        s, d = (k[0] + k[1]) / 4, (k[0] - k[1]) / 4
        self.K = [[s, d, -s], [d, s, -d], [-s, -d, s + k[2]]]
        q = hh / (self.a2 * k)
        self.G = [-q[0] - q[1] - q[2], -q[0] + q[1], -q[2]]
        self.om = [1 / p["tau_f"], 1 / (0.5 + p["M_phi"]), 1 / (0.5 + p["M_psi"])]

    def at(self, X, e):
        """X(r + e) at every r (periodic); axes of X are z, y, x."""
        n = [(-e[a], 2 - a) for a in range(3) if e[a]]
        return torch.roll(X, [s for s, _ in n], [d for _, d in n]) if n else X

    def ghosts(self, X):
        if self.solid is None:
            return X
        fluid = (~self.solid).to(F64)
        sums = []
        for axis in (True, False):
            es = [e for e in self.E if sum(map(abs, e)) == (1 if axis else 2)]
            sums.append((sum(self.at(fluid, e) for e in es), [sum(self.at(fluid * x, e) for e in es) for x in X]))
        (na, sa), (nd, sd) = sums
        out = []
        for c in range(3):
            ga = sa[c] / na.clamp(min=1) - self.G[c]
            gd = sd[c] / nd.clamp(min=1) - math.sqrt(2.0) * self.G[c]
            ghost = torch.where(na > 0, ga, torch.where(nd > 0, gd, torch.zeros_like(ga)))
            out.append(torch.where(self.solid, ghost, X[c]))
        return out

    def derivs(self, X):
        grad, lap = [], []
        for x in X:
            g, l = [0.0] * 3, 0.0
            for e, w in zip(self.E[1:], self.W[1:]):
                v = self.at(x, e)
                for a in range(3):
                    if e[a]:
                        g[a] = g[a] + 3 * w * e[a] * v
                l = l + 6 * w * (v - x)
            grad.append(g)
            lap.append(l)
        return grad, lap

    def tensor(self, e, a, b):
        """Weight of the gradient term G_ab of direction e."""
        if a != b:
            return e[a] * e[b] / 12
        on = e[a] != 0
        if sum(map(abs, e)) == 1:
            return (1 / 9 if on else -1 / 18) if self.dim == 2 else (5 / 36 if on else -1 / 9)
        return -1 / 72 if self.dim == 2 or on else 1 / 36

    def thermo(self, X, grad, lap):
        rho, phi, psi = X
        C = [(rho + phi - psi) / 2, (rho - phi - psi) / 2, psi]
        lC = [(lap[0] + lap[1] - lap[2]) / 2, (lap[0] - lap[1] - lap[2]) / 2, lap[2]]
        mu = [self.k[m] * (C[m] * (1 - C[m]) * (1 - 2 * C[m]) - self.a2 * lC[m]) for m in range(3)]
        pb = sum(self.k[m] / 2 * C[m] ** 2 * (1 - C[m]) * (1 - 3 * C[m]) for m in range(3))  # p_b - rho / 3
        L = sum(self.K[a][b] * X[a] * lap[b] for a in range(3) for b in range(3))
        D = self.dim
        Gab = {(a, b): sum(self.K[x][y] * grad[x][a] * grad[y][b] for x in range(3) for y in range(3))
               for a in range(D) for b in range(a, D)}
        return pb, L, Gab, (mu[0] - mu[1]) / 2, mu[2] - (mu[0] + mu[1]) / 2

    def force(self, pb, L, Gab):
        D = self.dim
        iso = pb - self.a2 * (sum(Gab[a, a] for a in range(D)) / 2 + L)
        P = {ab: self.a2 * g + (iso if ab[0] == ab[1] else 0.0) for ab, g in Gab.items()}
        F = [0.0] * D
        for e, w in zip(self.E[1:], self.W[1:]):
            for ab, v in P.items():
                for a, b in {ab, ab[::-1]}:
                    if e[b]:
                        F[a] = F[a] - 3 * w * e[b] * self.at(v, e)
        return F

    def equilibria(self, X, j):
        """Equilibria [3][Q] of the fields X and momentum j, and per direction the Guo source."""
        rho, phi, psi = X
        grad, lap = self.derivs(self.ghosts(X))
        pb, L, Gab, mp, ms = self.thermo(X, grad, lap)
        D = self.dim
        F = self.force(pb, L, Gab) if self.guo else None
        u = [(j[a] + (F[a] / 2 if F else 0.0)) / rho for a in range(D)]
        uu = sum(v * v for v in u)
        out, src = [[None] * len(self.E) for _ in range(3)], [None] * len(self.E)
        for i, (e, w) in enumerate(zip(self.E, self.W)):
            eu = sum(e[a] * u[a] for a in range(D) if e[a]) + 0.0 * rho
            if F:
                eF = sum(e[a] * F[a] for a in range(D) if e[a]) + 0.0 * rho
                src[i] = (1 - self.om[0] / 2) * w * (3 * (eF - sum(u[a] * F[a] for a in range(D))) + 9 * eu * eF)
            if i == 0:
                continue
            poly = 3 * eu + 4.5 * eu * eu - 1.5 * uu
            if self.guo:
                out[0][i] = w * rho * (1 + poly)
            else:
                out[0][i] = w * (rho + 3 * pb - 3 * self.a2 * L + rho * poly) + \
                    3 * self.a2 * sum(self.tensor(e, a, b) * g for (a, b), g in Gab.items() if self.tensor(e, a, b))
            out[1][i] = w * (3 * mp + phi * poly)
            out[2][i] = w * (3 * ms + psi * poly)
        for s in range(3):
            out[s][0] = X[s] - sum(out[s][1:])
        return out, src

    def moments(self, F):
        X = [sum(F[s]) for s in range(3)]
        j = [sum(e[a] * f for e, f in zip(self.E, F[0]) if e[a]) for a in range(self.dim)]
        if self.solid is not None:
            X = [torch.where(self.solid, torch.ones_like(X[0]) if s == 0 else torch.zeros_like(X[0]), X[s]) for s in range(3)]
        return X, j

    def start(self, X, u=None):
        if self.solid is not None:
            X = [torch.where(self.solid, torch.ones_like(X[0]), X[0]), X[1], X[2]]
        return self.equilibria(X, [X[0] * u[a] if u is not None else 0.0 * X[0] for a in range(self.dim)])[0]

    def step(self, F):
        X, j = self.moments(F)
        eq, src = self.equilibria(X, j)
        out = [[None] * len(self.E) for _ in range(3)]
        post = [[F[s][i] + self.om[s] * (eq[s][i] - F[s][i]) + (src[i] if self.guo and s == 0 else 0.0)
                 for i in range(len(self.E))] for s in range(3)]
        for i, e in enumerate(self.E):
            back = tuple(-c for c in e)
            for s in range(3):
                v = self.at(post[s][i], back)
                out[s][i] = v if self.solid is None or i == 0 else torch.where(self.at(self.solid, back), post[s][self.opp[i]], v)
        return out

    def fields(self, F):
        X, j = self.moments(F)
        C = [(X[0] + X[1] - X[2]) / 2, (X[0] - X[1] - X[2]) / 2, X[2]]
        if self.solid is not None:
            C = [torch.where(self.solid, torch.zeros_like(c), c) for c in C]
        return C, X[0], [v / X[0] for v in j]


def _flat(t):
    return t.detach().reshape(-1).cpu()


def exact(case, seed):
    if case["kind"] == "sweep":
        each = []
        for k in range(case["count"]):
            p, X, _, solid = _well(k, seed, case["nmax"])
            m = _Exact(p, solid)
            F = m.start(X)
            for _ in range(case["steps"]):
                F = m.step(F)
            each.append(m.fields(F)[0])
        return {"C%d" % (m + 1): torch.cat([_flat(c[m]) for c in each]) for m in range(3)}
    p, X, u, solid = _problem(case, seed)
    if case["kind"] == "inverse":
        target = X[2] + torch.where(solid, torch.zeros_like(X[2]), _uniform(seed + 77, *X[2].shape, lo=-0.03, hi=0.03))
        leaves = [torch.tensor(p["kappa"], dtype=F64, device="cuda"), torch.tensor(p["h"], dtype=F64, device="cuda")] + \
            [x.clone() for x in X]
        leaves = [t.requires_grad_(True) for t in leaves]
        m = _Exact(p, solid, leaves[0], leaves[1])
        F = m.start(leaves[2:])
        n = len(m.E)
        for _ in range(case["steps"]):
            # one step's intermediates at a time: the state alone is kept
            flat = checkpoint(
                lambda *a: tuple(sum((x for x in _Exact(p, solid, a[0], a[1]).step([list(a[2 + s * n:2 + (s + 1) * n]) for s in range(3)])), [])),
                leaves[0], leaves[1], *sum(F, []), use_reentrant=False)
            F = [list(flat[s * n:(s + 1) * n]) for s in range(3)]
        loss = ((m.fields(F)[0][2] - torch.where(solid, torch.zeros_like(target), target)) ** 2).sum()
        loss.backward()
        g = [t.grad for t in leaves]
        g[2:] = [torch.where(solid, torch.zeros_like(t), t) for t in g[2:]]
        return {"loss": loss.detach().cpu(), **{n: _flat(t) for n, t in zip(("kappa", "h", "rho", "phi", "psi"), g)}}
    m = _Exact(p, solid)
    with torch.no_grad():
        F = m.start(X, u)
        for _ in range(case["steps"]):
            F = m.step(F)
        C, rho, v = m.fields(F)
    out = {"C%d" % (m + 1): _flat(C[m]) for m in range(3)}
    if case["kind"] == "job":
        out["rho"] = _flat(rho)
        out["u"] = torch.stack([_flat(v[a]) if a < len(v) else torch.zeros(out["rho"].numel(), dtype=F64) for a in range(3)])
    return out
