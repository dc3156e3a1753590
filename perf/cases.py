"""What a user of this framework has it do, as timed cases: Split-Euler-Maruyama
steps of confined suspensions (one system or an ensemble), mobility, Stokes and
adjoint solves, the saddle matvec and the fluctuating forcing, through the
public entry points of the binding and the autograd function.

Sizes are those of the workloads, the tests and the benchmark, or generic.
exact() restates the method in plain 64-bit torch (matrix-free operator,
projection-preconditioned GMRES to 1e-13).  Lengths are in grid spacings.
"""
import math
import os

os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")   # as the benchmark sets it for ensembles

import numpy as np
import torch

import paper_1901_06427_gb300.binding as B
import workloads
from paper_1901_06427_gb300.autograd import MobilitySolve

KT, SEED_MASK = 1.0, (1 << 31) - 1


# ------------------------------------------------------------------ the cases
def _case(name, kind, setup, n=(0, 0, 0), **kw):
    c = {"name": name, "kind": kind, "setup": setup, "nx": n[0], "ny": n[1], "nz": n[2], "bodies": 0, "blobs": 12,
         "kernel": 3, "refined": False, "rtol": 1e-8, "periodic_x": False, "periodic_y": False, "free_top": False,
         "wall_speed": 0.0, "single": False, "systems": 0}
    c.update(kw)
    return c


def listed():
    return [
        # the tight two-sphere cavity at its coarsest resolution: the smallest step, all latency
        _case("step cavity 16x8x8", "step", "cavity", bodies=2, blobs=12, kernel=6, rtol=1e-10),
        # the two-sphere cavity of the benchmark: the ordinary step, FP64
        _case("step two spheres 48x48x32", "step", "two_sphere", bodies=2, blobs=42),
        # the same box with the six-point kernel, FP32 inside FP64 refinement: several restart cycles a solve
        _case("step six-point refined", "step", "two_sphere", bodies=2, blobs=42, kernel=6, refined=True,
              rtol=1e-10),
        # one boomerang in a doubly periodic slit: an axis longer than 48 points, many blobs per kernel width
        _case("step boomerang 64x64x16", "step", "boomerang", bodies=1, blobs=15, kernel=6, periodic_x=True,
              periodic_y=True, rtol=1e-11),
        # the driven monolayer: thin channel, moving wall, 1024 spheres, FP32 refined
        _case("step monolayer 384x96x12", "step", "monolayer", (64, 16, 12), bodies=1024, refined=True,
              periodic_x=True, wall_speed=0.5, rtol=1e-10),
        # an equilibrium ensemble: independent boxes of 16 to 48 points per axis, advanced together
        _case("ensemble of 24", "batch", "ensemble", refined=True, systems=24, rtol=1e-9),
        # one sphere's mobility at a tight tolerance, whole solution returned
        _case("mobility 32x32x32", "solve", "spheres", (32, 32, 32), bodies=1, blobs=42, rtol=1e-10),
        # unconstrained Stokes flow on a ragged box (no axis can be halved)
        _case("stokes 45x37x29", "stokes", "empty", (45, 37, 29), rtol=1e-10),
        # gradient of the mobility solve of 64 active spheres, forward and backward
        _case("gradient 128x128x64", "gradient", "spheres", (128, 128, 64), bodies=64, blobs=42, refined=True,
              rtol=1e-12),
        # the saddle matvec at memory-bound size in FP32, and in FP64 at an odd middling size
        _case("matvec f32 256x256x256", "matvec", "spheres", (256, 256, 256), bodies=64, blobs=42, single=True),
        _case("matvec f64 100x90x76", "matvec", "spheres", (100, 90, 76), bodies=8, blobs=42),
        # the fluctuating stress and its divergence
        _case("forcing 128x128x64", "forcing", "empty", (128, 128, 64)),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "solve", "stokes", "gradient", "matvec", "matvec", "forcing"])
    if kind == "batch":
        return _drawn(kind, "ensemble", refined=rng.random() < 0.6, systems=_size(rng, 2, 20), rtol=1e-9)
    if kind == "step" and rng.random() < 0.25:
        return _drawn(kind, "monolayer", (_size(rng, 6, 60), _size(rng, 2, 15), rng.choice([10, 12, 14, 16])),
                      refined=rng.random() < 0.6, periodic_x=True, wall_speed=rng.uniform(0.0, 0.6), rtol=1e-10)
    hi = {"step": 72, "solve": 80, "stokes": 96, "gradient": 64, "matvec": 220, "forcing": 120}[kind]
    n = tuple(_size(rng, 14, hi) for _ in range(3))
    if kind not in ("matvec", "forcing"):   # long axes are chosen so that they can be halved twice
        n = tuple(m if m <= 48 else 4 * (m // 4) for m in n)
    c = _drawn(kind, "empty" if kind in ("stokes", "forcing") else "spheres", n, refined=rng.random() < 0.4,
               periodic_x=rng.random() < 0.25, periodic_y=rng.random() < 0.15, free_top=rng.random() < 0.15,
               kernel=6 if rng.random() < 0.3 else 3, blobs=rng.choice([12, 12, 42]))
    if c["setup"] == "spheres":
        gap, wall = (7.0, 4.5) if c["blobs"] == 42 else (4.5, 3.0)
        c["bodies"] = rng.randint(1, min(24, int(np.prod([max(1, int((m - 2 * wall) // gap) + 1) for m in n]))))
        if kind == "step" and not c["free_top"]:
            c["wall_speed"] = rng.choice([0.0, 0.0, 0.4])
    c["rtol"] = 1e-12 if kind == "gradient" else 1e-10
    c["single"] = kind == "matvec" and rng.random() < 0.5
    return c


def _drawn(*args, **kw):
    c = _case("", *args, **kw)
    del c["name"]
    return c


# ----------------------------------------------------- a case as a workload
def _quats(rng, count):
    q = rng.standard_normal((count, 4))
    return q / np.linalg.norm(q, axis=1, keepdims=True)


def _spheres(case, rng):
    """Shells at random sites of a lattice with room for their jitter."""
    n = np.array([case["nx"], case["ny"], case["nz"]], dtype=float)
    radius, gap, wall = (2.5, 7.0, 4.5) if case["blobs"] == 42 else (1.0, 4.5, 3.0)
    count = np.maximum(1, ((n - 2 * wall) // gap).astype(int) + 1)
    sites = rng.permutation(int(count.prod()))[:case["bodies"]]
    pitch = np.where(count > 1, (n - 2 * wall) / np.maximum(count - 1, 1), 0.0)
    at = np.stack(np.unravel_index(sites, count), axis=1)
    q = np.where(count > 1, wall + at * pitch, n / 2) + rng.uniform(-0.4, 0.4, (len(sites), 3))
    shell = workloads.icosahedral_shell(case["blobs"], radius)
    w = workloads.Workload(name="spheres", n=tuple(int(v) for v in n))
    w.bodies = [workloads.Body(shell, q[i], t) for i, t in enumerate(_quats(rng, len(sites)))]
    w.potentials = {"gravity": 1.0, "pair_soft": {"phi0": 4.0, "b": 0.1 * radius, "d": 2.0 * radius},
                    "wall_soft": {"phi0": 4.0, "b": 0.1 * radius, "d": radius}}
    return w


def _workload(case, seed):
    """The workload of a case with bodies placed and turned from the seed."""
    rng = np.random.default_rng([int(seed) & SEED_MASK, 7])
    setup = case["setup"]
    if setup == "two_sphere":
        w = workloads.two_sphere_cavity(steps=1, kernel=case["kernel"])
    elif setup == "cavity":
        w = workloads.two_sphere_msd(case["blobs"])
    elif setup == "boomerang":
        w = workloads.boomerang_slit()
    elif setup == "monolayer":
        w = workloads.driven_monolayer(wall_speed=case["wall_speed"], cols=case["nx"], rows=case["ny"], nz=case["nz"],
                                       z=case["nz"] / 2)
    elif setup == "spheres":
        w = _spheres(case, rng)
    else:
        w = workloads.Workload(name="empty", n=(case["nx"], case["ny"], case["nz"]))
    if setup not in ("spheres", "empty"):
        turn = _quats(rng, w.n_bodies)
        if setup == "boomerang":          # the slit is lower than the boomerang is long: it turns about z
            turn = np.stack([np.cos(turn[:, 0]), 0 * turn[:, 0], 0 * turn[:, 0], np.sin(turn[:, 0])], axis=1)
        w.bodies = [workloads.Body(b.ref_blobs, b.q + rng.uniform(-0.05, 0.05, 3), turn[i])
                    for i, b in enumerate(w.bodies)]
    else:
        w.periodic = (bool(case["periodic_x"]), bool(case["periodic_y"]), False)
        w.free_slip = (False,) * 5 + (bool(case["free_top"]),)
        w.wall_vel = np.zeros((6, 3))
        w.wall_vel[5, 0] = case["wall_speed"]
    w.kernel = case["kernel"]
    w.rtol = case["rtol"]
    w.seed = int(rng.integers(1, 1 << 40))
    w.force_torque = rng.standard_normal((w.n_bodies, 6))
    slip = 0.1 * rng.standard_normal((w.n_blobs, 3))
    for a, b in zip(w.blob_offsets[:-1], w.blob_offsets[1:]):
        slip[a:b] -= slip[a:b].mean(axis=0)
    w.slip = slip
    return w


def _ensemble(case, seed):
    """Boxes and sphere counts of the ensemble workload, every body moved and turned from the seed."""
    out = []
    for i, w in enumerate(workloads.batched_ensemble(case["systems"])):
        rng = np.random.default_rng([int(seed) & SEED_MASK, 11, i])
        turn = _quats(rng, w.n_bodies)
        w.bodies = [workloads.Body(b.ref_blobs, b.q + rng.uniform(-0.1, 0.1, 3), turn[k]) for k, b in enumerate(w.bodies)]
        w.rtol, w.seed = case["rtol"], int(rng.integers(1, 1 << 40))
        out.append(w)
    return out


def _precision(case):
    return B.FP32_REFINED if case["refined"] else B.FP64


def _dev(x, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(x).ravel(), dtype=dtype, device="cuda")


def _random_field(case, seed, count):
    g = torch.Generator(device="cuda").manual_seed(int(seed) & SEED_MASK)
    return torch.randn(count, dtype=torch.float32 if case["single"] else torch.float64, device="cuda", generator=g)


# ------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "step": 1}
    if kind == "batch":
        ws = _ensemble(case, seed)
        s["grid"] = B.Batch(ws, precision=_precision(case))
        s["params"] = [B.sem_params(w.potentials, dt=w.dt, kT=KT) for w in ws]
        s["q"], s["quat"] = [_dev(w.q) for w in ws], [_dev(w.quat) for w in ws]
        s["seed"] = [w.seed for w in ws]
        return s
    w = _workload(case, seed)
    g = s["grid"] = B.grid_for(w, precision=_precision(case))
    s["seed"] = w.seed
    if kind == "step":
        s["params"] = B.sem_params(w.potentials, dt=w.dt, kT=KT)
        s["q"], s["quat"] = _dev(w.q), _dev(w.quat)
    elif kind in ("solve", "gradient"):
        s["FT"], s["slip"] = _dev(w.force_torque), _dev(w.slip)
        if kind == "gradient":
            s["r"] = g.blob_positions().requires_grad_(True)
            s["slip"].requires_grad_(True)
    elif kind == "stokes":
        s["f"] = _random_field(case, seed, g.layout()[3])
    elif kind == "matvec":
        s["x"] = _random_field(case, seed, g.n_total)
    return s


def run(state):
    s, g, kind = state, state["grid"], state["kind"]
    if kind == "batch":
        g.sem_step(s["params"], s["seed"], s["step"], s["q"], s["quat"])
        s["step"] += 1
        return [s["q"], s["quat"]]
    if kind == "step":
        g.sem_step(s["params"], s["seed"], s["step"], 0, s["q"], s["quat"])
        s["step"] += 1
        return [s["q"], s["quat"]]
    if kind == "solve":
        U, _, x = g.mobility_solve(s["FT"], slip=s["slip"], return_x=True)
        return [U, x]
    if kind == "gradient":
        U = MobilitySolve.apply(s["r"], s["slip"], g, s["FT"])
        return [U.detach(), *torch.autograd.grad((U ** 2).sum(), (s["r"], s["slip"]))]
    if kind == "stokes":
        v, pi, _ = g.stokes_solve(s["f"])
        return [v, pi]
    if kind == "matvec":
        return [g.apply_saddle(s["x"])]
    return [g.stochastic_forcing(KT, 0.05, s["seed"], s["step"])]


def work(case):
    """Solves: the right-hand side read, the solution written and the operator applied once; a step has three of
    them and draws the stress (nine normals a cell)."""
    if case["kind"] == "batch":
        ws = workloads.batched_ensemble(case["systems"])
        parts = [work(dict(case, kind="step", setup="spheres", nx=w.n[0], ny=w.n[1], nz=w.n[2], bodies=w.n_bodies))
                 for w in ws]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    n = {"two_sphere": (48, 48, 32), "boomerang": (64, 64, 16), "cavity": (16, 8, 8),
         "monolayer": (6 * case["nx"], 6 * case["ny"], case["nz"])}.get(case["setup"], (case["nx"], case["ny"], case["nz"]))
    bodies = case["nx"] * case["ny"] if case["setup"] == "monolayer" else case["bodies"]
    cells, blobs = float(np.prod(n)), bodies * case["blobs"]
    unknowns = 4 * cells + 3 * blobs + 6 * bodies
    once = {"bytes": 16 * unknowns, "flops": 36 * cells + 2 * 2 * 3 * case["kernel"] ** 3 * blobs}
    if case["single"]:
        once["bytes"] /= 2
    forcing = {"bytes": 8 * 3 * cells, "flops": 9 * cells * 30 + 3 * cells * 10}
    times = {"step": (3, 1), "gradient": (2, 0), "forcing": (0, 1)}.get(case["kind"], (1, 0))
    return {k: times[0] * once[k] + times[1] * forcing[k] for k in ("bytes", "flops")}


# ------------------------------------------------------- the method in 64 bits
def _six(r):
    """phi(r + 2 - t), t = 0..5, of the six-point kernel for r in [0, 1): its even and odd sums are 1/2, its moments
    0, 59/60 - sqrt(29)/20, 0, and phi(-3) = 0."""
    s = math.sqrt(29.0)
    beta = -7 / 3 * r ** 3 - 1.5 * r ** 2 + (9 + 7 * s) / 20 * r + (31 + 3 * s) / 40
    gamma = 5 / 72 * r ** 6 + (1 / 32 - s / 48) * r ** 4
    t = -2 * gamma / (beta + torch.sqrt(beta ** 2 - 112 * gamma))
    odd, even = (13 - s) / 80 * r, (7 + s) / 40 * r
    c = 29 / 480 - s / 160
    return torch.stack([-r ** 3 / 12 + r ** 2 / 8 - odd + c + t, r ** 3 / 6 - even + 0.25 - 3 * t,
                        -r ** 2 / 4 + 91 / 240 + s / 80 + 2 * t, -r ** 3 / 6 + even + 0.25 + 2 * t,
                        r ** 3 / 12 + r ** 2 / 8 + odd + c - 3 * t, t], dim=-1)


def _three(d):
    """phi(-1 - d), phi(-d), phi(1 - d) of the three-point kernel for d in [-1/2, 1/2)."""
    mid = (1 + torch.sqrt(1 - 3 * d ** 2)) / 3
    return torch.stack([(1 - mid - d) / 2, mid, (1 - mid + d) / 2], dim=-1)


class _Exact:
    """Saddle operator, right-hand sides and solves of one workload in 64-bit torch; fields are (z, y, x)."""

    def __init__(self, w):
        self.w, self.dev = w, "cuda"
        self.n, self.per, self.eta = w.n, w.periodic, w.eta
        self.shape = [[w.n[ax] - (ax == a and not w.periodic[ax]) for ax in (2, 1, 0)] for a in range(3)]
        self.cells = [w.n[2], w.n[1], w.n[0]]
        self.sizes = [int(np.prod(s)) for s in self.shape] + [int(np.prod(self.cells)), 3 * w.n_blobs, 6 * w.n_bodies]
        self.ghost = [[1.0 if f else -1.0 for f in w.free_slip[2 * ax:2 * ax + 2]] for ax in range(3)]
        self.vel = np.asarray(w.wall_vel)
        self.off = torch.as_tensor(w.blob_offsets, device=self.dev).long()
        self.body = torch.repeat_interleave(torch.arange(w.n_bodies, device=self.dev), self.off[1:] - self.off[:-1])
        self.ref = torch.as_tensor(w.ref_blobs, device=self.dev, dtype=torch.float64).reshape(-1, 3)
        self.bases = None
        if w.n_bodies:
            self.place(*(torch.as_tensor(v, device=self.dev) for v in (w.q, w.quat)))

    # bodies
    def place(self, q, quat):
        self.q, self.quat = q, quat
        self.arm = self.arms(quat)
        self.r = q[self.body] + self.arm
        self.table, self.lift = self.stencils(self.r)

    def arms(self, quat):
        u, s, v = quat[self.body, 1:], quat[self.body, :1], self.ref
        t = 2 * torch.linalg.cross(u, v)
        return v + s * t + torch.linalg.cross(u, t)

    def axis(self, a, ax, x):
        """Indices and folded weights of the kernel points along one axis, and twice the tangential wall speed that
        a ghost takes up (None on periodic axes and for the normal component)."""
        n, k = self.n[ax], self.w.kernel
        s = x - (0.0 if ax == a else 0.5)
        first = torch.floor(s.detach()) - 2 if k == 6 else torch.floor(s.detach() + 0.5) - 1
        wt = _six(s - first - 2) if k == 6 else _three(s - first - 1)
        p = first.long()[:, None] + torch.arange(k, device=self.dev)
        if self.per[ax]:
            return p % n, wt, None, None
        if ax == a:
            m = torch.where(p < 0, -p, torch.where(p > n, 2 * n - p, p))
            sign = torch.where((p < 0) | (p > n), -1.0, 1.0) * ((m >= 1) & (m <= n - 1))
            return (m - 1).clamp(0, n - 2), wt * sign, None, torch.where((p < 0) | (p > n), -1.0, 1.0)
        m = torch.where(p < 0, -1 - p, torch.where(p > n - 1, 2 * n - 1 - p, p))
        lo, hi = self.ghost[ax]
        sign = torch.where(p < 0, lo, torch.where(p > n - 1, hi, 1.0))
        speed = torch.where(p < 0, 2 * self.vel[2 * ax, a], torch.where(p > n - 1, 2 * self.vel[2 * ax + 1, a], 0.0))
        return m.clamp(0, n - 1), wt * sign, wt * speed, sign

    def stencils(self, r):
        """Per component: flat face index and weight of every kernel point, and what moving walls add to J v."""
        table, lift = [], []
        for a in range(3):
            (ix, wx, _, _), (iy, wy, _, _), (iz, wz, _, _) = A = [self.axis(a, ax, r[:, ax]) for ax in range(3)]
            e = self.shape[a]
            idx = ix[:, None, None, :] + e[2] * (iy[:, None, :, None] + e[1] * iz[:, :, None, None])
            wt = wz[:, :, None, None] * wy[:, None, :, None] * wx[:, None, None, :]
            table.append((idx.reshape(len(r), -1), wt.reshape(len(r), -1)))
            # folds act in x, y, z order: a later fold's wall speed carries the signs of the earlier ones
            part = torch.zeros(len(r), dtype=torch.float64, device=self.dev)
            for ax in range(3):
                if A[ax][2] is None:
                    continue
                f = A[ax][2].sum(1)
                for o in range(3):
                    if o != ax:
                        plain = A[o][1] if A[o][3] is None or o < ax else A[o][1] * A[o][3]
                        f = f * plain.sum(1)
                part = part + f
            lift.append(part)
        return table, torch.stack(lift, 1)

    def interp(self, v, table=None):
        return torch.stack([(f.reshape(-1)[i] * wt).sum(1) for f, (i, wt) in zip(v, table or self.table)], 1)

    def spread(self, lam, table=None):
        out = []
        for a, (i, wt) in enumerate(table or self.table):
            f = torch.zeros(self.sizes[a], dtype=torch.float64, device=self.dev)
            out.append(f.index_add_(0, i.reshape(-1), (wt * lam[:, a:a + 1]).reshape(-1)).reshape(self.shape[a]))
        return out

    def rigid(self, U, arm):
        return U[self.body, :3] + torch.linalg.cross(U[self.body, 3:], arm)

    def total(self, lam, arm):
        both = torch.cat([lam, torch.linalg.cross(arm, lam)], 1)
        return torch.zeros(self.w.n_bodies, 6, dtype=torch.float64, device=self.dev).index_add_(0, self.body, both)

    # fluid
    def split(self, x):
        p = torch.split(x, self.sizes[:len(self.sizes) if x.numel() > sum(self.sizes[:4]) else 4])
        v = [p[a].reshape(self.shape[a]) for a in range(3)]
        return (v, p[3].reshape(self.cells), *([p[4].reshape(-1, 3), p[5].reshape(-1, 6)] if len(p) > 4 else []))

    def join(self, *blocks):
        flat = []
        for b in blocks:
            flat += [f.reshape(-1) for f in b] if isinstance(b, list) else [b.reshape(-1)]
        return torch.cat(flat)

    def viscous(self, a, u):
        out = 6.0 * u
        for ax in range(3):
            d = 2 - ax
            if self.per[ax]:
                out = out - u.roll(1, d) - u.roll(-1, d)
                continue
            m = u.shape[d]
            out.narrow(d, 1, m - 1).sub_(u.narrow(d, 0, m - 1))
            out.narrow(d, 0, m - 1).sub_(u.narrow(d, 1, m - 1))
            if ax != a:
                out.narrow(d, 0, 1).sub_(self.ghost[ax][0] * u.narrow(d, 0, 1))
                out.narrow(d, m - 1, 1).sub_(self.ghost[ax][1] * u.narrow(d, m - 1, 1))
        return self.eta * out

    def grad(self, p):
        return [p - p.roll(1, 2 - a) if self.per[a] else p.diff(dim=2 - a) for a in range(3)]

    def div(self, v):
        out = 0.0
        for a in range(3):
            d = 2 - a
            if self.per[a]:
                out = out + v[a].roll(-1, d) - v[a]
            else:
                z = torch.zeros_like(v[a].narrow(d, 0, 1))
                out = out + torch.cat([v[a], z], d) - torch.cat([z, v[a]], d)
        return out

    def apply(self, x):
        v, p, *rest = self.split(x)
        f = [self.viscous(a, v[a]) + g for a, g in enumerate(self.grad(p))]
        if not rest:
            return self.join(f, -self.div(v))
        lam, U = rest
        if self.w.n_bodies:
            f = [a - b for a, b in zip(f, self.spread(lam))]
            return self.join(f, -self.div(v), self.rigid(U, self.arm) - self.interp(v), self.total(lam, self.arm))
        return self.join(f, -self.div(v))

    # preconditioner: exact viscous and pressure solves, free-space blob mobility of each body
    def basis(self, n, kind):
        T = 2 * torch.eye(n, dtype=torch.float64) - torch.diag(torch.ones(n - 1, dtype=torch.float64), 1)
        T = T - torch.diag(torch.ones(n - 1, dtype=torch.float64), -1)
        if kind == "periodic":
            T[0, n - 1] -= 1
            T[n - 1, 0] -= 1
        elif kind is not None:
            T[0, 0] -= kind[0]
            T[n - 1, n - 1] -= kind[1]
        lam, Q = torch.linalg.eigh(T)
        return lam.to(self.dev), Q.to(self.dev)

    def build(self):
        self.bases = []
        for g in range(4):
            kinds = ["periodic" if self.per[ax] else (1.0, 1.0) if g == 3 else None if ax == g else self.ghost[ax]
                     for ax in range(3)]
            e = self.cells if g == 3 else self.shape[g]
            self.bases.append([self.basis(e[2 - ax], kinds[ax]) for ax in range(3)])
        if self.w.n_bodies:
            self.blocks = []
            for p in range(self.w.n_bodies):
                s = slice(int(self.off[p]), int(self.off[p + 1]))
                self.blocks.append((s, torch.linalg.inv(self.rpy(self.r[s]))))

    def rpy(self, r):
        a = 1.47 if self.w.kernel == 6 else 0.91
        d = r[:, None] - r[None]
        s = d.norm(dim=2) + torch.eye(len(r), device=self.dev, dtype=torch.float64)
        far = s >= 2 * a
        c = 1 / (6 * math.pi * self.eta * a)
        one = torch.where(far, (1 + 2 * a * a / (3 * s * s)) * 0.75 * a / s, 1 - 9 * s / (32 * a)) * c
        two = torch.where(far, (1 - 2 * a * a / (s * s)) * 0.75 * a / s, 3 * s / (32 * a)) * c
        one.fill_diagonal_(c)
        M = one[:, :, None, None] * torch.eye(3, device=self.dev, dtype=torch.float64)
        M = M + (two / (s * s))[:, :, None, None] * d[..., :, None] * d[..., None, :]
        return M.permute(0, 2, 1, 3).reshape(3 * len(r), 3 * len(r))

    def invert(self, g, f):
        (lx, Qx), (ly, Qy), (lz, Qz) = self.bases[g]
        c = torch.einsum("zyx,xi,yj,zk->kji", f, Qx, Qy, Qz)
        lam = lz[:, None, None] + ly[:, None] + lx
        c = c / torch.where(lam > 1e-11, lam, torch.inf)
        return torch.einsum("kji,xi,yj,zk->zyx", c, Qx, Qy, Qz) / (1.0 if g == 3 else self.eta)

    def precondition(self, x):
        f, p, *rest = self.split(x)
        v = [self.invert(a, f[a]) for a in range(3)]
        q = p + self.div(v)
        phi = self.invert(3, q)
        v = [a + b for a, b in zip(v, self.grad(phi))]
        if not rest or not self.w.n_bodies:
            return self.join(v, -self.eta * q)
        s, U = rest[0] + self.interp(v), torch.empty_like(rest[1])
        lam = torch.empty_like(s)
        for b, (at, Mi) in enumerate(self.blocks):
            arm = self.arm[at]
            eye = torch.eye(3, dtype=torch.float64, device=self.dev).expand(len(arm), 3, 3)
            spin = torch.stack([torch.linalg.cross(e.expand_as(arm), arm) for e in eye[0]], 2)
            K = torch.cat([eye, spin], 2).reshape(-1, 6)
            t = Mi @ s[at].reshape(-1)
            U[b] = torch.linalg.solve(K.T @ Mi @ K, rest[1][b] + K.T @ t)
            lam[at] = (Mi @ (K @ U[b]) - t).reshape(-1, 3)
        return self.join(v, -self.eta * q, lam, U)

    def solve(self, b, tol=1e-13, most=400, cycle=120):
        """Flexible GMRES with two Gram-Schmidt passes; the pressure's mean is zero."""
        if self.bases is None:
            self.build()
        x, goal, done = torch.zeros_like(b), tol * float(b.norm()), 0
        while done < most:
            r = b - self.apply(x) if done else b
            beta = float(r.norm())
            if beta <= goal:
                break
            m = min(cycle, most - done)
            V, Z = torch.empty(m + 1, len(b), dtype=b.dtype, device=b.device), []
            V[0] = r / beta
            H = torch.zeros(m + 1, m, dtype=b.dtype)
            for j in range(m):
                Z.append(self.precondition(V[j]))
                u = self.apply(Z[j])
                for _ in range(2):
                    h = V[:j + 1] @ u
                    u = u - h @ V[:j + 1]
                    H[:j + 1, j] += h.cpu()
                H[j + 1, j] = float(u.norm())
                V[j + 1] = u / H[j + 1, j].item()
                done += 1
                e = torch.zeros(j + 2, 1, dtype=b.dtype)
                e[0] = beta
                y = torch.linalg.lstsq(H[:j + 2, :j + 1], e).solution
                if float((H[:j + 2, :j + 1] @ y - e).norm()) <= 0.3 * goal:
                    break
            for z, c in zip(Z, y[:, 0].tolist()):
                x = x + c * z
        v, p, *rest = self.split(x)
        return self.join(v, p - p.mean(), *rest)

    def rhs(self, FT=None, slip=None, fluid=None, walls=True):
        f = fluid or [torch.zeros(s, dtype=torch.float64, device=self.dev) for s in self.shape]
        if walls:
            for a in range(3):
                for ax in range(3):
                    if ax != a and not self.per[ax]:
                        d = 2 - ax
                        f[a].narrow(d, 0, 1).add_(2 * self.eta * self.vel[2 * ax, a])
                        f[a].narrow(d, f[a].shape[d] - 1, 1).add_(2 * self.eta * self.vel[2 * ax + 1, a])
        lam = (self.lift if walls else torch.zeros_like(self.r)) - (0.0 if slip is None else slip)
        return self.join(f, torch.zeros(self.cells, dtype=torch.float64, device=self.dev), lam, FT)

    # noise
    def normals(self, seed, step, purpose, count):
        """Box-Muller normals of the Philox4x64-10 blocks with key (seed, 0) and counter (block, step, purpose, 0)."""
        counter = ((purpose << 128) + (step << 64) - 1) % (1 << 256)   # numpy counts up before its first block
        words = np.random.Philox(counter=counter, key=seed).random_raw(4 * -(-count // 4))
        u = torch.as_tensor(((words >> np.uint64(12)) * np.uint64(2) + np.uint64(1)).astype(np.float64) * 2.0 ** -53)
        u = u.to(self.dev).reshape(-1, 2)
        rad, ang = torch.sqrt(-2 * torch.log(u[:, 0])), 2 * math.pi * u[:, 1]
        return torch.stack([rad * torch.cos(ang), rad * torch.sin(ang)], 1).reshape(-1)[:count]

    def forcing(self, dt, seed, step):
        shapes = {}
        for a in range(3):
            for b in (a, *(o for o in range(3) if o != a)):
                e = list(self.cells)
                if b != a:
                    e[2 - a] = self.shape[a][2 - a]
                    e[2 - b] = self.n[b] + (not self.per[b])
                shapes[a, b] = e
        z = torch.split(self.normals(seed, step, 1, sum(int(np.prod(e)) for e in shapes.values())),
                        [int(np.prod(e)) for e in shapes.values()])
        W = {k: t.reshape(e) for t, (k, e) in zip(z, shapes.items())}
        out = []
        for a in range(3):
            f = W[a, a] - W[a, a].roll(1, 2 - a) if self.per[a] else W[a, a].diff(dim=2 - a)
            for b in range(3):
                if b == a:
                    continue
                t, d = W[a, b].clone(), 2 - b
                if self.per[b]:
                    f = f + t.roll(-1, d) - t
                    continue
                for end, at in ((0, 0), (1, t.shape[d] - 1)):
                    t.narrow(d, at, 1).mul_(math.sqrt(2.0) if self.ghost[b][end] < 0 else 0.0)
                f = f + t.diff(dim=d)
            out.append(math.sqrt(2 * self.eta * KT / dt) * f)
        return out

    # one Split-Euler-Maruyama step
    def forces(self, pot):
        q, L = self.q, torch.tensor([float(m) for m in self.n], device=self.dev, dtype=torch.float64)
        F = torch.zeros(len(q), 6, dtype=torch.float64, device=self.dev)

        def soft(s, p):
            return p["phi0"] / p["b"] * torch.where(s < p["d"], torch.ones_like(s), torch.exp((p["d"] - s) / p["b"]))

        d = q[:, None] - q[None]
        for a in range(3):
            if self.per[a]:
                d[..., a] -= L[a] * torch.round(d[..., a] / L[a])
        s = d.norm(dim=2).fill_diagonal_(torch.inf)
        mag = torch.zeros_like(s)
        if "pair_soft" in pot:
            mag = mag + soft(s, pot["pair_soft"])
        if "yukawa" in pot:
            y = pot["yukawa"]
            mag = mag + y["u0"] * y["d_h"] * torch.exp((y["d_h"] - s) / y["lambda_d"]) * (1 / (y["lambda_d"] * s) + 1 / s ** 2)
        F[:, :3] += ((mag / s)[..., None] * d).sum(1)
        F[:, 2] -= pot.get("gravity", 0.0)
        f = torch.zeros_like(self.r)
        f[:, 2] -= pot.get("blob_gravity", 0.0)
        for a in range(3):
            if self.per[a]:
                continue
            if "wall_soft" in pot:
                F[:, a] += soft(q[:, a], pot["wall_soft"]) - soft(L[a] - q[:, a], pot["wall_soft"])
            if "blob_wall_soft" in pot:
                f[:, a] += soft(self.r[:, a], pot["blob_wall_soft"]) - soft(L[a] - self.r[:, a], pot["blob_wall_soft"])
        F += self.total(f, self.arm)
        if "substrate" in pot:
            c = 4 * math.pi / (math.sqrt(3.0) * pot["substrate"]["s_lattice"])
            X = torch.stack([q[:, 0], q[:, 1] - L[1] / 2], 1)
            k1, k2 = (torch.tensor([-c * math.sqrt(3.0) / 2, v * c / 2], device=self.dev, dtype=torch.float64) for v in (-1, 1))
            for k in (k1 - k2, k1, k2):
                F[:, :2] -= 0.5 * pot["substrate"]["u0"] * torch.sin(X @ k)[:, None] * k
        return F

    def turn(self, quat, phi):
        ang = phi.norm(dim=1, keepdim=True)
        u = phi * torch.where(ang > 0, torch.sin(ang / 2) / ang, torch.full_like(ang, 0.5))
        c, s, v = torch.cos(ang / 2), quat[:, :1], quat[:, 1:]
        out = torch.cat([c * s - (u * v).sum(1, keepdim=True), c * v + s * u + torch.linalg.cross(u, v)], 1)
        return out / out.norm(dim=1, keepdim=True)

    def sem_step(self, dt, pot, seed, step):
        nb, delta = self.w.n_bodies, 2.0 ** (-52.0 / 3.0)
        F, slip = self.forces(pot), 0.0
        W = self.normals(seed, step, 2, 6 * nb).reshape(nb, 6)
        length = torch.stack([torch.cdist(*[self.ref[self.off[p]:self.off[p + 1]]] * 2).max() for p in range(nb)])[:, None]
        v, _, lam, U = self.split(self.solve(self.rhs(KT * torch.cat([W[:, :3] / length, W[:, 3:]], 1), walls=False)))
        sharp = [torch.zeros_like(f) for f in v]
        for sign in (1.0, -1.0):
            quat = self.turn(self.quat, 0.5 * sign * delta * W[:, 3:])
            arm = self.arms(quat)
            table, _ = self.stencils((self.q + 0.5 * sign * delta * length * W[:, :3])[self.body] + arm)
            sharp = [f + sign / delta * g for f, g in zip(sharp, self.spread(lam, table))]
            F = F - sign / delta * self.total(lam, arm)
            slip = slip + sign / delta * (self.rigid(U, arm) - self.interp(v, table))
        both = self.join(sharp, torch.zeros(self.cells, dtype=torch.float64, device=self.dev))
        slip = slip - self.interp(self.split(self.solve(both))[0])
        x = self.solve(self.rhs(F, slip, self.forcing(dt, seed, step)))
        U = self.split(x)[3]
        return (self.q + dt * U[:, :3]).reshape(-1), self.turn(self.quat, dt * U[:, 3:]).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        new = [_Exact(w).sem_step(w.dt, w.potentials, w.seed, 1) for w in _ensemble(case, seed)]
        return [[q for q, _ in new], [t for _, t in new]]
    w = _workload(case, seed)
    E = _Exact(w)
    if kind == "step":
        return list(E.sem_step(w.dt, w.potentials, w.seed, 1))
    if kind == "forcing":
        return [E.join(E.forcing(0.05, w.seed, 1))]
    if kind == "stokes":
        f = _random_field(case, seed, sum(E.sizes[:3]))
        v, p = E.split(E.solve(torch.cat([f, f.new_zeros(E.sizes[3])])))
        return [E.join(v), p.reshape(-1)]
    if kind == "matvec":
        return [E.apply(_random_field(case, seed, sum(E.sizes)).double())]
    FT, slip = (torch.as_tensor(t, device=E.dev, dtype=torch.float64) for t in (w.force_torque, w.slip))
    x = E.solve(E.rhs(FT, slip))
    v, _, lam, U = E.split(x)
    if kind == "solve":
        return [U.reshape(-1), x]
    # gradient of sum U^2: the transposed system has the same operator, with the forces 2 U
    z, _, mu, V = E.split(E.solve(E.rhs(2 * U, walls=False)))
    r = E.r.clone().requires_grad_(True)
    arm = r - E.q[E.body]
    table, _ = E.stencils(r)
    value = (lam * E.interp(z, table)).sum() + (mu * E.interp(v, table)).sum()
    value = value - (mu * E.rigid(U, arm)).sum() - (V * E.total(lam, arm)).sum()
    return [U.reshape(-1), torch.autograd.grad(value, r)[0].reshape(-1), -mu.reshape(-1)]
