"""The flow computations users of this framework run, as cases to time.

A case is one workload at one size: a refined periodic box, the channel, the
flow past a sphere, the Rayleigh-Benard cell, or the gradient through a
periodic box.  ``run`` advances it by a few coarse steps and reads the
macroscopic fields of every patch, as a simulation's output loop does (the
gradient case takes the objective and its gradient).  ``exact`` restates the
method in plain torch at 64 bits.

Sizes: the full and reduced forms of the workloads the framework is configured
for, ordinary ones between them, and odd extents, where rows do not end on a
tile, a vector or a power of two.
"""
import itertools
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1608_06915_gb300 import lbm

T0 = 1.0 / 3.0


# ---------------------------------------------------------------------------
# the cases

def _box(name, nx, ny, nz, refined, storage, steps, autotune, nu=0.01):
    return dict(name=name, kind="box", nx=nx, ny=ny, nz=nz, refined=refined, storage=storage, steps=steps,
                autotune=autotune, nu=nu)


def _channel(name, nx, ny, nz, storage, steps, autotune):
    return dict(name=name, kind="channel", nx=nx, ny=ny, nz=nz, storage=storage, steps=steps, autotune=autotune)


def _sphere(name, scale, nx, ny, nz, curved, storage, steps, autotune):
    return dict(name=name, kind="sphere", scale=scale, nx=nx, ny=ny, nz=nz, curved=curved, storage=storage,
                steps=steps, autotune=autotune)


def _rbc(name, nx, ny, nz, l1, l2, pr, storage, steps, autotune):
    return dict(name=name, kind="rbc", nx=nx, ny=ny, nz=nz, l1=l1, l2=l2, pr=pr, storage=storage, steps=steps,
                autotune=autotune)


def _gradient(name, n, steps, every, storage, autotune):
    return dict(name=name, kind="gradient", nx=n, ny=n, nz=n, refined=True, steps=steps, every=every,
                storage=storage, autotune=autotune, nu=0.01)


def listed():
    return [
        # the smallest call: one step of a small uniform box and its fields, as a
        # coupled or interactive program takes it; launches and latency
        _box("box_uniform_24", 24, 24, 24, False, "fp32", 1, False),
        # the two-level Taylor-Green validation run, in the precision it is validated in
        _box("tgv_32_fp64", 32, 32, 32, True, "fp64", 10, False),
        # a two-level box at an ordinary size, a run of steps between outputs
        _box("box_refined_64", 64, 64, 64, True, "fp32", 20, True),
        # a uniform box with odd rows, no refinement: the plain lattice Boltzmann use
        _box("box_uniform_odd", 149, 131, 117, False, "fp32", 4, True),
        # the gradient of the kinetic energy, one checkpoint per 20 steps
        _gradient("gradient_64", 64, 40, 20, "fp32", True),
        # the three-level channel at full size, plain and 16-bit storage
        _channel("channel_fp32", 256, 64, 128, "fp32", 4, True),
        _channel("channel_fp16", 256, 64, 128, "fp16s", 4, True),
        # a channel of the user's own extents
        _channel("channel_odd", 101, 49, 75, "fp32", 4, True),
        # the four-level sphere at full size: large coarse level, small fine ones,
        # inlet, outlet, solid nodes
        _sphere("sphere_fp32", 0, 384, 192, 192, False, "fp32", 4, True),
        # the reduced sphere with its curved surface: many small launches per step
        _sphere("sphere_curved_48", 1, 48, 24, 24, True, "fp32", 4, False),
        # the three-level Rayleigh-Benard cell at full size (two population sets)
        _rbc("rbc_fp32", 256, 256, 128, 12, 6, 0.7, "fp32", 2, True),
        # a small cell of the other Prandtl regime, odd sides, double precision
        _rbc("rbc_pr2_fp64", 37, 22, 32, 8, 4, 2.0, "fp64", 4, False),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["box", "box", "channel", "channel", "sphere", "rbc", "gradient"])
    tune = rng.random() < 0.7
    if kind == "box":
        n = [log(24, 200) for _ in range(3)]
        storage = rng.choice(["fp32", "fp32", "fp16s", "bf16s", "fp64"])
        c = _box("", *n, rng.random() < 0.6, storage, rng.randint(1, 10), tune, round(rng.uniform(0.002, 0.05), 4))
    elif kind == "channel":
        n = log(16, 256), rng.randint(32, 64), log(8, 128)
        c = _channel("", *n, rng.choice(["fp32", "fp32", "fp16s", "bf16s", "fp64"]), rng.randint(1, 4), tune)
    elif kind == "sphere":
        s = rng.randint(1, 3)
        n = 48 * s + rng.randint(0, 96), 24 * s + rng.randint(0, 24), 24 * s + rng.randint(0, 24)
        c = _sphere("", s, *n, rng.random() < 0.5, rng.choice(["fp32", "fp32", "fp16s", "bf16s"]), rng.randint(1, 4),
                    tune)
    elif kind == "rbc":
        fp64 = rng.random() < 0.25
        top = 48 if fp64 else 200
        l2 = rng.randint(4, 6)
        n = log(8, top), log(8, top), rng.randint(4 * l2 + 16, 64 if fp64 else 128)
        c = _rbc("", *n, 2 * l2, l2, rng.choice([0.25, 0.7, 2.0, 4.0]), "fp64" if fp64 else "fp32", rng.randint(1, 2),
                 tune)
    else:
        every = rng.choice([5, 10, 20])
        c = _gradient("", rng.randint(24, 64), every * rng.randint(1, 2), every, rng.choice(["fp32", "fp32", "fp64"]),
                      tune)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# the workloads: the description lbm.Grid takes, and the initial fields

def _bands(n, axis, l1, l2):
    """Refinement bands of levels 1 and 2 along both walls of an axis."""
    top = [k - 1 for k in n]
    out = []
    for lev, width in ((1, l1), (2, l2)):
        for low in (True, False):
            lo, hi = [0, 0, 0], list(top)
            if low:
                hi[axis] = width
            else:
                lo[axis] = top[axis] - width
            out.append((lev, tuple(lo), tuple(hi)))
    return out


def problem(case):
    n = (case["nx"], case["ny"], case["nz"])
    p = dict(name=case["kind"], n=n, periodic=(1, 1, 1), walls=(0,) * 6, inflow_axis=-1, u_in=(0, 0, 0), boxes=[],
             solid=None, nu0=case.get("nu", 0.01), accel0=(0, 0, 0), mirror_lbgk=False, thermal=None)
    if case["kind"] in ("box", "gradient"):
        if case["refined"]:
            # a centred box of about half the width, at least 8 spacings
            lo = tuple(min(3 * k // 8, (k - 8) // 2) if case["kind"] == "gradient" else k // 4 for k in n)
            p["boxes"] = [(1, lo, tuple(k - a for k, a in zip(n, lo)))]
    elif case["kind"] == "channel":
        height, u_tau = n[1] - 0.75, 0.0045
        p.update(periodic=(1, 0, 1), walls=(0, 0, 1, 1, 0, 0), boxes=_bands(n, 1, 8, 4),
                 nu0=u_tau * height / 2 / 180.0, accel0=(2 * u_tau * u_tau / height, 0, 0))
    elif case["kind"] == "sphere":
        s = case["scale"]
        if s == 0:
            boxes = [(1, (80, 80, 80), (160, 112, 112)), (2, (86, 86, 86), (132, 106, 106)),
                     (3, (90, 89, 89), (110, 103, 103))]
            centre, d = (96.0, 96.0, 96.0), 64.0
        else:
            boxes = [(lev, tuple(s * v for v in lo), tuple(s * v for v in hi)) for lev, lo, hi in
                     ((1, (8, 4, 4), (36, 20, 20)), (2, (10, 6, 6), (30, 18, 18)), (3, (12, 8, 8), (24, 16, 16)))]
            centre, d = (18.0 * s, 12.0 * s, 12.0 * s), 24.0 * s
        lo = [int(8 * c - d / 2) - 1 for c in centre]
        ax = [np.arange(a, a + int(d) + 3) - 8 * c for a, c in zip(lo, centre)]
        r2 = ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2
        p.update(periodic=(0, 1, 1), inflow_axis=0, u_in=(0.05, 0.0, 0.0), boxes=boxes, nu0=0.05 * d / 3700.0 / 8.0,
                 solid=dict(level=3, lo=tuple(lo), mask=(r2 < d * d / 4).astype(np.uint8)))
        if case["curved"]:
            p["wall_shape"] = dict(kind="sphere", c=centre, r=d / 16.0, solid_inside=True)
    else:
        height, dt, u_ff = n[2] - 0.75, 0.01, 0.05
        p.update(periodic=(1, 1, 0), walls=(0, 0, 0, 0, 1, 1), boxes=_bands(n, 2, case["l1"], case["l2"]),
                 nu0=u_ff * height * math.sqrt(case["pr"] / 1e7) if n[2] > 64 else 0.01,
                 thermal=dict(pr=case["pr"], t0=T0, glambda=u_ff * u_ff / (dt * height), t_ref=T0, dT=dt,
                              wall_T=(0, 0, 0, 0, T0 + dt / 2, T0 - dt / 2)))
    return p


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _dtype(case):
    return torch.float64 if case["storage"] == "fp64" else torch.float32


def _noise(shape, seed, patch):
    g = torch.Generator(device=_device())
    g.manual_seed(1000003 * int(seed) + patch)
    return 2.0 * torch.rand(shape, generator=g, device=_device(), dtype=torch.float32).double() - 1.0


def fields(case, prob, seed, patch, level, org, dim):
    """rho, u and (thermal) T, float64 values of the case's precision, over a box
    of nodes of one patch."""
    h = 1.0 / (1 << level)
    x, y, z = (((torch.arange(d, device=_device(), dtype=torch.float64) + o) * h).reshape(
        [-1 if 2 - a == k else 1 for k in range(3)]) for a, (o, d) in enumerate(zip(org, dim)))
    shape = tuple(reversed(dim))
    noise = _noise((3,) + shape, seed, patch)
    n = prob["n"]
    T = None
    if case["kind"] == "gradient":
        # a smooth solenoidal field of a few large modes
        r = np.random.RandomState(seed % (1 << 31))
        u = torch.zeros((3,) + shape, device=_device(), dtype=torch.float64)
        for _ in range(12):
            k = r.randint(-3, 4, 3)
            k[r.randint(3)] = r.randint(1, 4)
            a = np.cross(k, r.normal(size=3)) / np.linalg.norm(k)
            ph = sum(2 * math.pi * int(k[b]) / n[b] * (x, y, z)[b] for b in range(3)) + float(r.uniform(0, 2 * math.pi))
            for b in range(3):
                u[b] += 0.012 * float(a[b]) * torch.cos(ph)
    elif case["kind"] == "box":
        # Taylor-Green vortex with a little noise
        u = 0.0005 * noise
        kx, ky = 2 * math.pi / n[0], 2 * math.pi / n[1]
        u[0] += 0.05 * torch.sin(kx * x) * torch.cos(ky * y)
        u[1] -= 0.05 * torch.cos(kx * x) * torch.sin(ky * y)
    elif case["kind"] == "channel":
        # laminar profile with 5% perturbations
        height = n[1] - 0.75
        prof = 0.42 * (y + 0.125) * (height - y - 0.125) / height ** 2
        u = 0.05 * noise * prof
        u[0] += prof
    elif case["kind"] == "sphere":
        u = 0.0005 * noise
        u[0] += 0.05
    else:
        # convection rolls between the plates, 1% temperature noise
        th, height = prob["thermal"], n[2] - 0.75
        zeta, k = (z + 0.125) / height, 2 * math.pi / n[0]
        u = 0.0002 * noise
        u[0] -= 0.02 * torch.sin(k * x) * torch.cos(math.pi * zeta) * torch.sin(math.pi * zeta)
        u[2] += 0.02 * torch.cos(k * x) * torch.sin(math.pi * zeta) ** 2
        T = T0 + th["dT"] * (0.5 - zeta + 0.2 * torch.cos(k * x) * torch.sin(math.pi * zeta) + 0.01 * noise[1])
        T = T.expand(shape).contiguous()
    out = torch.ones(shape, device=_device(), dtype=torch.float64), u, T
    return tuple(None if v is None else v.to(_dtype(case)).double() for v in out)


class _Patch:
    """One refinement box: region, faces toward the parent, parent hole."""

    def __init__(self, prob, level, lo, hi):
        n, self.level, self.kids, self.parent = prob["n"], level, [], -1
        s = 1 << level
        self.span = [bool(prob["periodic"][a]) and lo[a] == 0 and hi[a] == n[a] - 1 for a in range(3)]
        self.org = [0 if self.span[a] else s * lo[a] for a in range(3)]
        self.dim = [s * n[a] if self.span[a] else s * (hi[a] - lo[a]) + 1 for a in range(3)]
        self.flo = [level > 0 and not self.span[a] and not (lo[a] == 0 and prob["walls"][2 * a]) for a in range(3)]
        self.fhi = [level > 0 and not self.span[a] and not (hi[a] == n[a] - 1 and prob["walls"][2 * a + 1])
                    for a in range(3)]
        self.lo, self.hi = lo, hi
        self.blo, self.bhi = [s // 2 * v for v in lo], [s // 2 * v for v in hi]  # in parent coordinates

    def inset(self, a, k):
        """Range along axis a, parent coordinates, k nodes inside the interface faces."""
        return (self.blo[a] + k if self.flo[a] else -(1 << 40)), (self.bhi[a] - k if self.fhi[a] else 1 << 40)

    def volume(self, k):
        """Parent nodes k inside the interface faces (k = 2: the hole)."""
        v = 1
        for a in range(3):
            lo, hi = self.inset(a, k)
            v *= self.dim[a] // 2 if self.span[a] else min(hi, self.bhi[a]) - max(lo, self.blo[a]) + 1
        return v


def _patches(prob):
    n = prob["n"]
    out = [_Patch(prob, 0, (0, 0, 0), tuple(k - 1 for k in n))]
    for lev, lo, hi in sorted(prob["boxes"], key=lambda b: b[0]):
        c = _Patch(prob, lev, lo, hi)
        c.parent = next(q for q, p in enumerate(out) if p.level == lev - 1 and
                        all(p.lo[a] <= lo[a] and hi[a] <= p.hi[a] for a in range(3)))
        out[c.parent].kids.append(len(out))
        out.append(c)
    return out


def prepare(case, seed):
    prob = problem(case)
    grid = lbm.Grid(prob, case["storage"])
    boxes = _patches(prob)
    init = []
    for q, (p, info) in enumerate(zip(boxes, grid.patches)):
        rho, u, T = fields(case, prob, seed, q, p.level, p.org, p.dim)
        at = tuple(slice(info["org"][a] - p.org[a], info["org"][a] - p.org[a] + info["dim"][a]) for a in (2, 1, 0))
        init.append(tuple(None if v is None else v[(Ellipsis,) + at].to(_dtype(case)).contiguous()
                          for v in (rho, u, T)))
        grid.init_equilibrium(q, *init[-1])
    if case["autotune"]:
        grid.autotune(trials=2)
        for q, f in enumerate(init):
            grid.init_equilibrium(q, *f)
    state = dict(grid=grid, case=case, dtype=_dtype(case))
    if case["kind"] == "gradient":
        state["u0"] = [u.requires_grad_(True) for _, u, _ in init]
    return state


def run(state):
    grid, case = state["grid"], state["case"]
    if case["kind"] == "gradient":
        J = lbm.kinetic_energy_run(grid, state["u0"], case["steps"], case["every"])
        return [J.detach().to(state["dtype"])] + list(torch.autograd.grad(J, state["u0"]))
    grid.step(case["steps"])
    out = []
    for q in range(len(grid.patches)):
        rho, u, T, _ = grid.moments(q, dtype=state["dtype"])
        out.append([rho, u, T] if case["kind"] == "rbc" else [rho, u])
    return out


def work(case):
    prob = problem(case)
    boxes = _patches(prob)
    updates = nodes = 0
    for p in boxes:
        v = math.prod(p.dim) - sum(boxes[k].volume(2) for k in p.kids)
        if prob["solid"] is not None and prob["solid"]["level"] == p.level:
            v -= int(prob["solid"]["mask"].sum())
        nodes += v
        updates += v << p.level
    size = dict(fp64=8, fp32=4, fp16s=2, bf16s=2)[case["storage"]]
    sets = 2 if case["kind"] == "rbc" else 1
    if case["kind"] == "gradient":
        # forward: read and write the populations; reverse: read them and lambda, write lambda
        return dict(bytes=updates * case["steps"] * 5 * 27 * size + nodes * 3 * 16,
                    flops=updates * case["steps"] * 3400)
    out = nodes * (27 * sets * size + (4 + (sets > 1)) * (8 if size == 8 else 4))
    return dict(bytes=updates * case["steps"] * 54 * size * sets + out, flops=updates * case["steps"] * 850 * sets)


# ---------------------------------------------------------------------------
# the method in plain torch, 64 bits: populations [27, nodes], every node of a
# patch's region stored (hole nodes too, never read)

_C = np.array([[i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1] for i in range(27)])
_W = np.prod(np.where(_C == 0, 2.0 / 3.0, 1.0 / 6.0), axis=1)


def _const(a):
    return torch.tensor(a, dtype=torch.float64, device=_device())


def _feq(rho, u):
    s = torch.sqrt(1 + 3 * u * u)
    b = (2 * u + s) / (1 - u)
    A = 2 - s
    ax = [torch.stack([A[a] / b[a], 4 * A[a], A[a] * b[a]]) / 6 for a in range(3)]
    return (ax[2][:, None, None] * ax[1][None, :, None] * ax[0][None, None, :]).reshape(27, -1) * rho


def _macro(f):
    rho = f.sum(0)
    return rho, _const(_C.T) @ f / rho


def _collide(f, beta, du):
    """KBC collision; du [3, nodes] or None (exact difference method)."""
    rho, u = _macro(f)
    fe = _feq(rho, u)
    df = f - fe
    c = _C
    P = _const(np.stack([c[:, 0] ** 2, c[:, 1] ** 2, c[:, 2] ** 2, c[:, 0] * c[:, 1], c[:, 0] * c[:, 2],
                         c[:, 1] * c[:, 2]])) @ df
    dev = torch.cat([P[:3] - P[:3].mean(0), P[3:]])
    na = (c != 0).sum(1)
    face, edge = (na == 1)[:, None], (na == 2)[:, None]
    S = np.concatenate([0.5 * (face & (c != 0)), 0.25 * edge * np.stack(
        [c[:, 0] * c[:, 1], c[:, 0] * c[:, 2], c[:, 1] * c[:, 2]], 1)], 1)
    ds = _const(S) @ dev
    dh = df - ds
    sh, hh = (ds * dh / fe).sum(0), (dh * dh / fe).sum(0)
    ok = hh > 1e-30 * rho * rho
    gam = torch.where(ok, 1 / beta - (2 - 1 / beta) * sh / torch.where(ok, hh, torch.ones_like(hh)),
                      torch.full_like(hh, 2.0))
    if du is not None:
        fe = _feq(rho, u + du)
    return fe + (1 - beta * gam) * df + beta * (gam - 2) * ds


def _geq(rho, u, e):
    cu, c2 = _const(_C) @ u, _const((_C ** 2).sum(1))[:, None]
    u2 = (u * u).sum(0)
    return _const(_W)[:, None] * (e + 3 * (e + 2 * rho / 3) * cu +
                                  4.5 * ((e + 4 * rho / 3) * (cu * cu - u2 / 3) + 2 * rho / 9 * (c2 - 1)))


def _stress(f):
    return torch.stack([torch.stack([_const(_C[:, a] * _C[:, b]) @ f for b in range(3)]) for a in range(3)])


class _Exact:
    def __init__(self, case, seed):
        self.prob = prob = problem(case)
        self.P = _patches(prob)
        self.L = 1 + max(p.level for p in self.P)
        self.thermal = th = prob["thermal"]
        nu3 = 1.0 / (6.0 * prob["nu0"] + 1.0)
        al3 = 1.0 / (6.0 * prob["nu0"] / th["pr"] + 1.0) if th else nu3
        self.swap = bool(th) and th["pr"] > 1
        b, b1 = (al3, nu3) if self.swap else (nu3, al3)
        self.beta = []
        for _ in range(self.L):
            self.beta.append((b, b1))
            b, b1 = 1 / (1 + 2 * (1 / b - 1)), 1 / (1 + 2 * (1 / b1 - 1))
        self.init = [fields(case, prob, seed, q, p.level, p.org, p.dim) for q, p in enumerate(self.P)]
        for q, p in enumerate(self.P):
            self._layout(q, p)
        for q, p in enumerate(self.P):
            self._coupling(q, p)

    def _coords(self, p, idx):
        return [p.org[0] + idx % p.dim[0], p.org[1] + idx // p.dim[0] % p.dim[1],
                p.org[2] + idx // (p.dim[0] * p.dim[1])]

    def _layout(self, q, p):
        """Pull sources (27 flat indices per node), node classes."""
        prob, dev = self.prob, _device()
        nx, ny, nz = p.dim
        N = nx * ny * nz
        own = torch.arange(N, device=dev)
        maxc = [(prob["n"][a] - 1) << p.level for a in range(3)]
        solid = torch.zeros(N, dtype=torch.bool, device=dev)
        if prob["solid"] is not None and prob["solid"]["level"] == p.level:
            m = torch.tensor(prob["solid"]["mask"], device=dev, dtype=torch.bool)
            o = [prob["solid"]["lo"][a] - p.org[a] for a in range(3)]
            solid.view(nz, ny, nx)[o[2]:o[2] + m.shape[0], o[1]:o[1] + m.shape[1], o[0]:o[0] + m.shape[2]] = m
        p.N, p.tab, p.curved = N, torch.empty((27, N), dtype=torch.int64, device=dev), []
        for i in range(27):
            src, bounce = 0, torch.zeros((nz, ny, nx), dtype=torch.bool, device=dev)
            for a, stride in ((0, 1), (1, nx), (2, nx * ny)):
                k = torch.arange(p.dim[a], device=dev)
                s = k - int(_C[i, a])
                shape = [-1 if 2 - a == d else 1 for d in range(3)]
                if p.span[a]:
                    s = s % p.dim[a]
                elif not prob["periodic"][a]:
                    g = s + p.org[a]
                    wall = ((g < 0) & bool(prob["walls"][2 * a])) | ((g > maxc[a]) & bool(prob["walls"][2 * a + 1]))
                    bounce |= wall.reshape(shape)
                # beyond the outlet: the last node; beyond an interface: never read
                s = s.clamp(0, p.dim[a] - 1)
                src = src + (s * stride).reshape(shape)
            src, bounce = src.reshape(-1), bounce.reshape(-1)
            hit = solid[src] & ~solid
            p.tab[i] = torch.where(bounce | hit, (26 - i) * N + own, i * N + src)
            shape = prob.get("wall_shape")
            if shape is not None and bool(hit.any()):
                # the returning population interpolated along the link to the sphere
                at = own[hit]
                X = torch.stack(self._coords(p, at)).double() / (1 << p.level)
                step = -_const(_C[i])[:, None] / (1 << p.level)
                rel = X - _const(shape["c"])[:, None]
                qa, qb, qc = (step * step).sum(0), 2 * (step * rel).sum(0), (rel * rel).sum(0) - shape["r"] ** 2
                disc = qb * qb - 4 * qa * qc
                t = torch.where(disc >= 0, (-qb - torch.sqrt(disc.clamp(min=0))) / (2 * qa), torch.full_like(qb, -1.0))
                t = torch.where((t > 0) & (t <= 1), t, torch.full_like(t, 0.5))
                behind = at + int(_C[i, 0]) + nx * int(_C[i, 1]) + nx * ny * int(_C[i, 2])
                p.curved.append((i, at, behind, solid[behind], t))
        X = self._coords(p, own)
        exists = torch.ones(N, dtype=torch.bool, device=dev)
        p.cf = torch.zeros(N, dtype=torch.bool, device=dev)
        for k in p.kids:
            hole, twin = (self._inside(self.P[k], X, d) for d in (2, 1))
            exists &= ~hole
            p.cf |= twin & ~hole
        p.exists, p.solid, p.depth = exists, solid, torch.full((N,), 1 << 40, device=dev)
        for a in range(3):
            if p.flo[a]:
                p.depth = torch.minimum(p.depth, X[a] - p.org[a])
            if p.fhi[a]:
                p.depth = torch.minimum(p.depth, p.org[a] + p.dim[a] - 1 - X[a])
        p.inlet = own[(X[0] == 0) & ~solid] if p.level == 0 and prob["inflow_axis"] == 0 else None

    @staticmethod
    def _inside(c, X, k):
        """Parent nodes X at least k inside the interface faces of box c."""
        ok = torch.ones_like(X[0], dtype=torch.bool)
        for a in range(3):
            lo, hi = c.inset(a, k)
            ok &= (X[a] >= lo) & (X[a] <= hi)
        return ok

    def _local(self, p, X):
        out, stride = 0, 1
        for a in range(3):
            v = X[a]
            if self.prob["periodic"][a]:
                v = v % (self.prob["n"][a] << p.level)
            out = out + (v - p.org[a]) * stride
            stride *= p.dim[a]
        return out

    def _coupling(self, q, c):
        if c.level == 0:
            return
        par, dev = self.P[c.parent], _device()
        own = torch.arange(par.N, device=dev)
        X = self._coords(par, own)
        at = own[self._inside(c, X, 1) & ~self._inside(c, X, 2)]
        c.twin = at, self._local(c, [2 * v for v in self._coords(par, at)])
        c.target = torch.nonzero(c.depth <= 1).reshape(-1)

    # -- node maps: a state is (f,) or (f, g)
    def _stream(self, p, st):
        f = st[0]
        out = torch.take(f, p.tab)
        for i, at, behind, lost, t in p.curved:
            back, fwd = f[26 - i, at], f[i, at]
            mix = torch.where(lost, back, 2 * t * back + (1 - 2 * t) * f[26 - i, torch.where(lost, at, behind)])
            out[i, at] = torch.where(t < 0.5, mix, back / (2 * t) + (2 * t - 1) / (2 * t) * fwd)
        if not self.thermal:
            return (out,)
        g = torch.take(st[1], p.tab).reshape(27, p.dim[2], -1)
        rho = f.sum(0).reshape(p.dim[2], -1)
        for i in range(27):  # isothermal plates across z: anti-bounce-back
            for face, k, c in ((4, 0, 1), (5, p.dim[2] - 1, -1)):
                z = p.org[2] + k
                if _C[i, 2] == c and z == (0 if face == 4 else (self.prob["n"][2] - 1) << p.level):
                    tw = self.thermal["wall_T"][face]
                    g[i, k] = -g[i, k] + 2 * _W[i] * rho[k] * (3 * tw + int((_C[i] ** 2).sum()) - 1)
        return out, g.reshape(27, -1)

    def _moments(self, st):
        rho, u = _macro(st[0])
        if not self.thermal:
            return rho, u, None, None
        e = st[1].sum(0)
        return rho, u, e, (e / rho - (u * u).sum(0)) / 3

    def _relax(self, level, st):
        beta, beta1 = self.beta[level]
        rho, u, e, T = self._moments(st)
        if not self.thermal:
            du = [a / (1 << level) for a in self.prob["accel0"]]
            return (_collide(st[0], beta, _const(du)[:, None] if any(du) else None),)
        du = torch.zeros_like(u)
        du[2] = self.thermal["glambda"] / (1 << level) * (T - self.thermal["t_ref"])
        f = _collide(st[0], beta, du)
        P1 = _stress(st[0]) - rho * (u[:, None] * u[None] + torch.eye(3, device=u.device, dtype=u.dtype)[..., None] / 3)
        Pu = 2 * (P1 * u[None]).sum(1)
        X = Pu if self.swap else _const(_C.T) @ st[1] - (e + 2 * rho / 3) * u - Pu
        W = _const(_W)[:, None]
        if self.swap:
            cc = _const(np.einsum("ia,ib->iab", _C, _C) - np.eye(3) / 3).reshape(27, 9)
            f = f + 9 * (beta - beta1) * W * (cc @ P1.reshape(9, -1))
        g = st[1]
        return f, g + 2 * beta * (_geq(rho, u, e) - g) + 6 * (beta - beta1) * W * (_const(_C) @ X)

    def _collide_all(self, level, st):
        n, step = st[0].shape[1], 1 << 21
        if n <= step:
            return self._relax(level, st)
        for k in range(0, n, step):
            for x, y in zip(st, self._relax(level, tuple(x[:, k:k + step] for x in st))):
                x[:, k:k + step] = y
        return st

    def _neq(self, st, src, dst, r):
        """Moments and non-equilibrium parts rescaled from level src to dst, r = dx_src / dx_dst."""
        rho, u, e, T = self._moments(st)
        ff, fg = self.beta[src][0] / (r * self.beta[dst][0]), self.beta[src][1] / (r * self.beta[dst][1])
        if src == dst:
            ff = fg = 1.0
        if self.swap:
            ff, fg = fg, ff
        fn = st[0] - _feq(rho, u)
        if not self.thermal:
            return (rho, u), (ff * fn,)
        Y = 2 * (_stress(fn) * u[None]).sum(1)
        gn = fg * (st[1] - _geq(rho, u, e)) + (ff - fg) * 3 * _const(_W)[:, None] * (_const(_C) @ Y)
        return (rho, u, T), (ff * fn, gn)

    def _compose(self, m, neq):
        f = _feq(m[0], m[1]) + neq[0]
        if not self.thermal:
            return (f,)
        return f, _geq(m[0], m[1], m[0] * (3 * m[2] + (m[1] * m[1]).sum(0))) + neq[1]

    def _explode(self, c, pre_p, pre_c):
        """Interface nodes of a child: tensor four-point Lagrange interpolation."""
        par, w4 = self.P[c.parent], (-1 / 16, 9 / 16, 9 / 16, -1 / 16)
        Y = torch.stack(self._coords(c, c.target))
        out = [torch.empty((27, c.target.numel()), device=Y.device, dtype=torch.float64) for _ in pre_c]
        for mask in itertools.product((0, 1), repeat=3):
            at = torch.nonzero(((Y & 1) == torch.tensor(mask, device=Y.device)[:, None]).all(0)).reshape(-1)
            if not at.numel():
                continue
            acc = None
            for ks in itertools.product(*[range(4) if m else (None,) for m in mask]):
                S = [Y[a, at] // 2 if k is None else (Y[a, at] - 3 + 2 * k) // 2 for a, k in enumerate(ks)]
                w = math.prod(w4[k] for k in ks if k is not None)
                for a in range(3):
                    if self.prob["periodic"][a]:
                        S[a] = S[a] % (self.prob["n"][a] << par.level)
                child = self._inside(c, S, 1)
                zero = torch.zeros_like(at)
                ip = torch.where(child, zero, self._local(par, S))
                ic = torch.where(child, self._local(c, [2 * v for v in S]), zero)
                vp = self._neq(tuple(x[:, ip] for x in pre_p), par.level, c.level, 2.0)
                vc = self._neq(tuple(x[:, ic] for x in pre_c), c.level, c.level, 1.0)
                v = [w * torch.where(child, y, x) for x, y in zip(vp[0] + vp[1], vc[0] + vc[1])]
                acc = v if acc is None else [x + y for x, y in zip(acc, v)]
            k = len(acc) - len(pre_c)
            for o, y in zip(out, self._relax(c.level, self._compose(acc[:k], acc[k:]))):
                o[:, at] = y
        return out

    def step(self, F):
        for k in range(1, (1 << (self.L - 1)) + 1):
            active = [q for q, p in enumerate(self.P) if k % (1 << (self.L - 1 - p.level)) == 0]
            pre = {q: self._stream(self.P[q], F[q]) for q in active}
            # what the coupling reads of the pre-states, before they are collided
            coupled = {}
            for q in active:
                p, put = self.P[q], []
                for kid in p.kids:
                    c = self.P[kid]
                    at, src = c.twin
                    m, neq = self._neq(tuple(x[:, src] for x in pre[kid]), c.level, p.level, 0.5)
                    put.append((at, self._relax(p.level, self._compose(m, neq))))
                if p.level and p.parent in active:
                    put.append((p.target, self._explode(p, pre[p.parent], pre[q])))
                if p.inlet is not None:
                    put.append((p.inlet, tuple(x[:, p.inlet] for x in F[q])))
                coupled[q] = put
            F = list(F)
            for q in active:
                new = self._collide_all(self.P[q].level, pre.pop(q))
                for at, vals in coupled[q]:
                    new = tuple(x.index_copy(1, at, v) for x, v in zip(new, vals))
                F[q] = new
        return F

    def start(self, u=None):
        F = []
        for q, p in enumerate(self.P):
            rho, v, T = self.init[q]
            rho, v = rho.reshape(-1), (v if u is None else u[q]).reshape(3, -1)
            if p.inlet is not None:
                v = v.clone()
                v[:, p.inlet] = _const(self.prob["u_in"])[:, None]
            f = _feq(rho, v)
            if T is None:
                F.append((f,))
            else:
                F.append((f, _geq(rho, v, rho * (3 * T.reshape(-1) + (v * v).sum(0)))))
        return F

    def stored(self, p, x):
        """Values [.., N] on the bounding box of the patch's nodes, zero where there is no fluid."""
        m = p.exists.view(p.dim[2], p.dim[1], p.dim[0])
        at = []
        for d in range(3):
            low, high = (e for e in range(3) if e != d)
            k = torch.nonzero(m.any(dim=high).any(dim=low)).reshape(-1)
            at.append(slice(int(k[0]), int(k[-1]) + 1))
        x = torch.where(p.exists & ~p.solid, x, torch.zeros_like(x)).reshape(x.shape[:-1] + m.shape)
        return x[(Ellipsis,) + tuple(at)].contiguous()

    def outputs(self, F):
        out = []
        for p, st in zip(self.P, F):
            rho, u, _, T = self._moments(st)
            du = [a / (1 << p.level) for a in self.prob["accel0"]]
            u = u + 0.5 * _const(du)[:, None]
            if self.thermal:
                u[2] += 0.5 * self.thermal["glambda"] / (1 << p.level) * (T - self.thermal["t_ref"])
            out.append([self.stored(p, x) for x in ((rho, u, T) if self.thermal else (rho, u))])
        return out

    def energy(self, F):
        J = 0.0
        for p, (f,) in zip(self.P, F):
            own = p.exists & ~p.cf & (p.depth >= 2)
            rho, u = _macro(f)
            J = J + 0.5 * 0.125 ** p.level * torch.where(own, rho * (u * u).sum(0), torch.zeros_like(rho)).sum()
        return J


def exact(case, seed):
    e = _Exact(case, seed)
    if case["kind"] != "gradient":
        with torch.no_grad():
            F = e.start()
            for _ in range(case["steps"]):
                F = e.step(F)
            return e.outputs(F)
    u = [v.requires_grad_(True) for _, v, _ in e.init]
    F = e.start(u)

    def step(*flat):
        return tuple(x for (x,) in e.step([(x,) for x in flat]))

    flat = tuple(x for (x,) in F)
    for _ in range(case["steps"]):
        flat = checkpoint(step, *flat, use_reentrant=False)
    J = e.energy([(x,) for x in flat])
    grads = torch.autograd.grad(J, u)
    return [J.detach()] + [e.stored(p, g.reshape(3, -1)) for p, g in zip(e.P, grads)]
