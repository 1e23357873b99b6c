"""Workloads of the soft-body library, as a program that uses it runs them.

A case is a mesh family with its sizes, the material options in use and the
call that is made: an equilibrium layer forward and backward, one or several
backward-Euler steps with their backward, a checkpointed rollout with
backpropagation through time, a batch of bodies, or one of the element-level
maps.  Meshes are jittered grids (triangulated rectangles, boxes cut into 5 or
6 tets a hex) of any cell counts, numbered along the grid or in random order
as mesh generators leave them.

Solver tolerances are tight (1e-10 to 1e-12, as the accuracy comparisons of
this repository use): the results are then those of the physical problem to
well below 1e-9, whatever path the iterations took to them.
"""
import functools
import math

import numpy as np
import torch

from paper_2102_05791_gb300 import api

DEV = "cuda:0"
MU, LAM, K_MUSCLE, GRAVITY, DENSITY = 1.0e4, 4.0e4, 5.0e3, 9.8, 1.0e3
DT, K_CONTACT = 1.0 / 30.0, 1.0e6

BASE = dict(nz=0, split=0, precision="mixed", muscle=0, log_mode=0, friction=0.0, shuffle=False, steps=1, bodies=1)


def listed():
    def case(name, kind, **kw):
        return dict(BASE, name=name, kind=kind, **kw)

    return [
        # the smallest layer: a 256-triangle body inside a training loop, latency only
        case("equilibrium_2d_small", "quasi", nx=16, ny=8),
        # an ordinary soft body of a design problem: 40,960 tets, equilibrium + dL/da
        case("equilibrium_3d", "quasi", nx=32, ny=16, nz=16, split=5),
        # the same layer in FP64, ragged sizes, mesh-generator numbering, active-spring muscle
        case("equilibrium_3d_fp64", "quasi", nx=19, ny=11, nz=10, split=6, precision="fp64", muscle=1, shuffle=True),
        # a large body, 393,216 tets
        case("equilibrium_3d_large", "quasi", nx=64, ny=32, nz=32, split=6),
        # the largest: 3,145,728 tets, 1.6 M unknowns; the adjoint of a known state with every
        # parameter's gradient (muscle activations and material), as inverse design calls it
        case("adjoint_3d_largest", "adjoint", nx=128, ny=64, nz=64, split=6),
        # one control step of a tet body on the ground: backward-Euler with friction and its backward
        case("step_3d", "step", nx=13, ny=9, nz=8, split=6, friction=2.0e3, log_mode=1, shuffle=True),
        # the 64 x 32 walker: rollout and backpropagation through time
        case("walker_bptt", "rollout", nx=64, ny=32, steps=12),
        # many bodies of uneven size in one call (200 to 8,000 triangles each), rollout + BPTT
        case("batch_2d", "batch", nx=0, ny=0, bodies=256, steps=4),
        # a handful of small bodies, as a per-GPU shard of a population holds them
        case("batch_2d_few", "batch", nx=0, ny=0, bodies=12, steps=6),
        # element-level maps for a caller's own solver: H v and (E, grad E) of the largest body
        case("hvp_3d_largest", "hvp", nx=128, ny=64, nz=64, split=6),
        case("energy_grad_3d", "energy", nx=64, ny=32, nz=32, split=6),
        # H v of a small body: launches count
        case("hvp_2d_small", "hvp", nx=33, ny=17, shuffle=True),
    ]


def draw(rng):
    kind = rng.choice(["quasi", "quasi", "quasi", "adjoint", "step", "rollout", "batch", "hvp", "energy"])
    c = dict(BASE, kind=kind, shuffle=rng.random() < 0.4, log_mode=int(rng.random() < 0.25))
    dim = 3 if rng.random() < 0.6 else 2
    log_u = lambda lo, hi: math.exp(rng.uniform(math.log(lo), math.log(hi)))  # noqa: E731
    if kind == "batch":
        n = int(log_u(3, 256))
        return dict(c, nx=0, ny=0, bodies=n, steps=rng.randint(1, 4), shuffle=False, log_mode=0)
    if kind == "rollout":
        dim = 2
    if kind in ("step", "rollout"):
        c["friction"] = rng.choice([0.0, 2.0e3])
        c["steps"] = rng.randint(2, 10) if kind == "rollout" else 1
    if kind in ("quasi", "step"):
        c["muscle"] = int(rng.random() < 0.3)
        if rng.random() < 0.25:
            c["precision"] = "fp64"
    hi = {"quasi": 400e3, "adjoint": 1500e3, "step": 40e3, "rollout": 6e3, "hvp": 3000e3, "energy": 1500e3}[kind]
    if c["precision"] == "fp64":
        hi = min(hi, 40e3)
    if dim == 2:
        hi = min(hi, 100e3)
    n = log_u(250, hi)
    if dim == 2:
        ny = max(3, int(round(math.sqrt(n / 2.0 / 2.0) * rng.uniform(0.8, 1.1))))
        return dict(c, nx=max(3, int(n / 2.0 / ny)), ny=ny)
    split = rng.choice([5, 6])
    s = (n / split / 2.0) ** (1.0 / 3.0)
    ny = max(2, int(round(s * rng.uniform(0.85, 1.1))))
    nz = max(2, int(round(s * rng.uniform(0.8, 1.2))))
    return dict(c, nx=max(2, int(n / split / ny / nz)), ny=ny, nz=nz, split=split)


# ---------------------------------------------------------------- meshes

HEX5 = {0: [(0, 3, 5, 6), (1, 0, 3, 5), (2, 0, 3, 6), (4, 0, 5, 6), (7, 3, 5, 6)],
        1: [(1, 2, 4, 7), (0, 1, 2, 4), (3, 1, 2, 7), (5, 1, 4, 7), (6, 2, 4, 7)]}
HEX6 = [(0, 1, 3, 7), (0, 1, 5, 7), (0, 2, 3, 7), (0, 2, 6, 7), (0, 4, 5, 7), (0, 4, 6, 7)]


def grid(nx, ny, nz, split, rng, shuffle):
    """Rest positions X and elements T of a jittered grid of height 1 (2D when nz is 0);
    `low` marks the vertices of the bottom row or face.  Corner k of a hex has offsets
    (k & 1, k >> 1 & 1, k >> 2)."""
    dim = 3 if nz else 2
    n = np.array([nx, ny, nz][:dim])
    h = 1.0 / ny
    idx = np.stack(np.meshgrid(*[np.arange(k + 1) for k in n[::-1]], indexing="ij")[::-1], axis=-1).reshape(-1, dim)
    X = idx * h
    inner = ((idx > 0) & (idx < n)).all(axis=1)
    X = X + inner[:, None] * rng.uniform(-0.1, 0.1, size=X.shape) * h
    low = idx[:, 1] == 0
    cell = np.stack(np.meshgrid(*[np.arange(k) for k in n[::-1]], indexing="ij")[::-1], axis=-1).reshape(-1, dim)
    stride = np.cumprod(np.concatenate([[1], n[:-1] + 1]))
    base = cell @ stride
    corner = lambda k: base + sum(int(k >> c & 1) * int(stride[c]) for c in range(dim))  # noqa: E731
    if dim == 2:
        T = np.stack([np.stack([corner(k) for k in t], axis=1) for t in ((0, 1, 3), (0, 3, 2))], axis=1)
    elif split == 6:
        T = np.stack([np.stack([corner(k) for k in t], axis=1) for t in HEX6], axis=1)
    else:
        even, odd = [np.stack([np.stack([corner(k) for k in t], axis=1) for t in HEX5[q]], axis=1) for q in (0, 1)]
        T = np.where((cell.sum(axis=1) % 2 == 0)[:, None, None], even, odd)
    T = T.reshape(-1, dim + 1)
    bad = np.linalg.det(idx[T[:, 1:]] - idx[T[:, :1]]) < 0
    T[bad, 1], T[bad, 2] = T[bad, 2], T[bad, 1].copy()
    if shuffle:
        to = rng.permutation(len(X))
        at = np.argsort(to)
        X, low, T = X[at], low[at], to[T][rng.permutation(len(T))]
    return np.ascontiguousarray(X), np.ascontiguousarray(T.astype(np.int32)), low


class Body:
    """One mesh with its material and per-element inputs (host arrays).  The mesh belongs to the case
    (`shape` is its generator); fibers and all that a call takes come from the seed (`rng`)."""

    def __init__(self, case, shape, rng, nx=None, ny=None):
        dyn = case["kind"] in ("step", "rollout", "batch")
        self.X, self.T, low = grid(nx or case["nx"], ny or case["ny"], case["nz"], case["split"], shape, case["shuffle"])
        self.fixed = (low & (not dyn)).astype(np.uint8)
        g = rng.standard_normal((len(self.T), self.X.shape[1]))
        self.fiber = g / np.linalg.norm(g, axis=1, keepdims=True)
        self.mu = float(shape.uniform(5e3, 2e4)) if case["kind"] == "batch" else MU
        self.lam = 4.0 * self.mu
        self.k_muscle, self.density, self.gravity = K_MUSCLE, DENSITY, GRAVITY
        self.k_contact, self.contact_power = (K_CONTACT, 3) if dyn else (0.0, 3)
        self.dt = DT if dyn else 0.0
        self.k_friction, self.eps_friction = case["friction"], 0.01
        self.log_mode, self.muscle_model = case["log_mode"], case["muscle"]

    def simulator(self, case):
        return api.Simulator(self.X, self.T, self.fixed, self.fiber, mu=self.mu, lam=self.lam, k_muscle=self.k_muscle,
                             density=self.density, gravity=self.gravity, k_contact=self.k_contact,
                             contact_power=self.contact_power, log_mode=self.log_mode, dt=self.dt,
                             k_friction=self.k_friction, eps_friction=self.eps_friction,
                             muscle_model=self.muscle_model, precision=case["precision"], max_cg=2000, device=DEV,
                             **tolerances(case))


def tolerances(case):
    return dict(newton_rtol=1e-11, adjoint_rtol=1e-11)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), device=DEV)


def activations(case, n, rng, steps=0):
    """Muscle activations; over the steps of a rollout each element follows a 1 Hz sinusoid."""
    lo, hi = (0.6, 1.0) if case["muscle"] else (0.0, 1.0)
    if not steps:
        return rng.uniform(lo, hi, size=n)
    t = np.arange(steps)[:, None] * DT
    mid, amp = 0.5 * (lo + hi), 0.4 * (hi - lo)
    return mid + amp * np.sin(2.0 * math.pi * t + rng.uniform(0.0, 2.0 * math.pi, size=n))


def moved(X, amp, rng):
    """A deformed state: rest shape, a smooth field that vanishes on the bottom, a little noise."""
    dim = X.shape[1]
    s = X / X.max(axis=0)
    smooth = np.stack([np.sin(2.0 * s[:, (c + 1) % dim] + c) * s[:, 1] for c in range(dim)], axis=1)
    noise = rng.uniform(-1.0, 1.0, size=X.shape) * (X[:, 1:2] > 0.0)
    return X + amp * smooth + 0.02 * noise * spacing(X)


def spacing(X):
    return (np.prod(X.max(axis=0)) / len(X)) ** (1.0 / X.shape[1])


def inputs(case, seed):
    """The host arrays of a case: its bodies and what the call takes."""
    shape = np.random.default_rng([case["nx"], case["ny"], case["nz"], case["split"], case["bodies"]])
    rng = np.random.default_rng([seed, case["nx"], case["ny"], case["nz"], case["bodies"]])
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":
        bodies = []
        for _ in range(case["bodies"]):
            tris = math.exp(shape.uniform(math.log(200.0), math.log(8000.0)))
            ny = max(2, int(round(math.sqrt(tris / 4.0))))
            bodies.append(Body(case, shape, rng, nx=max(2, int(round(tris / 2.0 / ny))), ny=ny))
    else:
        bodies = [Body(case, shape, rng)]
    X = np.concatenate([b.X for b in bodies])
    ne = sum(len(b.T) for b in bodies)
    v = {"bodies": bodies, "X": X}
    if kind in ("quasi", "adjoint", "hvp", "energy"):
        v["a"] = activations(case, ne, rng)
        v["target"] = X.mean(axis=0) + rng.uniform(-0.1, 0.1, size=X.shape[1]) * X.max(axis=0)
    if kind in ("adjoint", "hvp", "energy"):
        v["x"] = moved(X, 0.02, rng)
    if kind == "adjoint":  # the gradient of a tracking loss on every vertex
        v["g"] = (moved(X, 0.03, rng) - v["x"]) / len(X)
        v["g"][bodies[0].fixed.astype(bool)] = 0.0
    if kind == "hvp":
        v["v"] = rng.standard_normal(X.shape)
    if kind in ("step", "rollout", "batch"):
        v["x0"] = X + np.array([0.0, 0.002, 0.0])[: X.shape[1]]
        v["v0"] = 0.1 * (moved(X, 1.0, rng) - X)
        v["a"] = activations(case, ne, rng, steps if kind != "step" else 0)
        v["gx"] = np.concatenate([np.tile(np.eye(X.shape[1])[0] / len(b.X), (len(b.X), 1)) for b in bodies])
        v["gv"] = 0.01 * rng.standard_normal(X.shape) / len(X)
    return v


def prepare(case, seed):
    v = inputs(case, seed)
    s = {k: dev(x) for k, x in v.items() if isinstance(x, np.ndarray)}
    s["case"] = case
    if case["kind"] == "batch":
        s["batch"] = api.Batch(v["bodies"], max_cg=2000, max_adjoint_cg=8000, threads=512, **tolerances(case))
    else:
        s["sim"] = v["bodies"][0].simulator(case)
    if case["kind"] == "hvp":
        s["v"] = s["v"].to(s["sim"].vec_dtype)
    return s


def run(s):
    kind, sim = s["case"]["kind"], s.get("sim")
    if kind == "quasi":
        a = s["a"].clone().requires_grad_(True)
        x = api.QuasistaticSolve.apply(sim, a)
        loss = 0.5 * (x.mean(dim=0) - s["target"]).square().sum()
        loss.backward()
        return {"x": x.detach(), "da": a.grad}
    if kind == "adjoint":
        lam, _ = sim.adjoint(s["x"], s["a"], s["g"])
        da = sim.param_vjp(s["x"], s["a"], lam)
        dmu, dlam, dk = sim.material_vjp(s["x"], s["a"], lam)
        return {"lam": lam, "da": da, "dmu": dmu, "dlam": dlam, "dk": dk}
    if kind == "hvp":
        return {"Hv": sim.hvp(s["x"], s["a"], s["v"])}
    if kind == "energy":
        E, g = sim.energy_grad(s["x"], s["a"])
        return {"E": E, "g": g}
    if kind == "batch":
        sx, sv, ab, xb, vb, _, mg = s["batch"].rollout(s["x0"], s["v0"], s["a"], s["gx"], s["gv"], material_grad=True)
        return {"x": sx, "v": sv, "da": ab, "dx0": xb, "dv0": vb, "dmat": mg}
    x0, v0, a = [s[k].clone().requires_grad_(True) for k in ("x0", "v0", "a")]
    if kind == "step":
        x1, v1 = api.BEStep.apply(sim, x0, v0, a)
    else:
        x1, v1 = api.Rollout.apply(sim, x0, v0, a, 4)
    torch.autograd.backward([x1, v1], [s["gx"], s["gv"]])
    return {"x": x1.detach(), "v": v1.detach(), "dx0": x0.grad, "dv0": v0.grad, "da": a.grad}


def sizes(case):
    """(vertices, elements) of a case; a batch's from the mean of its size distribution."""
    if case["kind"] == "batch":
        tris = case["bodies"] * (8000.0 - 200.0) / math.log(8000.0 / 200.0)
        return 0.55 * tris, tris
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if not nz:
        return (nx + 1) * (ny + 1), 2 * nx * ny
    return (nx + 1) * (ny + 1) * (nz + 1), case["split"] * nx * ny * nz


def work(case):
    """Inputs read once and outputs written once; for the solves, whose iteration counts belong to the
    method, the operations of one gradient and of one Hessian product a step and direction."""
    nv, ne = sizes(case)
    d = 3 if case["nz"] else 2
    kind, steps = case["kind"], case["steps"]
    mesh = ne * (4 * (d + 1) + 8 * d) + nv * 8 * d  # elements, fibers, rest positions
    hvp, grad = (470.0, 260.0) if d == 3 else (170.0, 100.0)
    if kind == "hvp":
        return {"bytes": mesh + ne * 8 + nv * d * (8 + 4 + 4), "flops": ne * hvp}
    if kind == "energy":
        return {"bytes": mesh + ne * 8 + nv * d * 16, "flops": ne * 1.5 * grad}
    if kind == "adjoint":
        return {"bytes": mesh + ne * 40 + nv * d * 24, "flops": ne * (hvp + grad)}
    if kind == "quasi":
        return {"bytes": mesh + ne * 16 + nv * d * 16, "flops": ne * (2 * hvp + grad)}
    return {"bytes": mesh + steps * ne * 16 + nv * d * 64 + (steps * nv * d * 16 if kind == "batch" else 0),
            "flops": steps * ne * (2 * hvp + grad)}


# ---------------------------------------------------------------- the same in 64 bits, in plain torch

class Exact:
    """The energy's derivatives and the solves in FP64 torch: element Hessians from automatic
    differentiation of the energy density, a dense factorisation for small bodies and conjugate
    gradients for the others."""

    def __init__(self, b):
        self.b, self.dim = b, b.X.shape[1]
        self.X, self.T, self.f = dev(b.X), dev(b.T.astype(np.int64)), dev(b.fiber)
        self.free = ~dev(b.fixed.astype(bool))
        D = (self.X[self.T[:, 1:]] - self.X[self.T[:, :1]]).transpose(1, 2)
        B = torch.linalg.inv(D)
        self.W = torch.linalg.det(D) / math.factorial(self.dim)
        self.S = torch.cat([-B.sum(dim=1, keepdim=True), B], dim=1)  # shape gradients [ne, corner, axis]
        self.mass = torch.zeros(len(self.X), dtype=torch.float64, device=DEV)
        self.mass.index_add_(0, self.T.reshape(-1),
                             (b.density * self.W / (self.dim + 1)).repeat_interleave(self.dim + 1))
        self.scale = b.dt * b.dt if b.dt > 0 else 1.0
        self.fw = torch.zeros_like(self.mass)

    def psi(self, F, f, a):
        b = self.b
        J = (F[0, 0] * F[1, 1] - F[0, 1] * F[1, 0] if self.dim == 2 else
             (F[:, 0] * torch.linalg.cross(F[:, 1], F[:, 2])).sum())
        ll = torch.log(J) if b.log_mode == 0 else (J - 1) - 0.5 * (J - 1) ** 2
        q2 = (F @ f).square().sum()
        m = 0.5 * b.k_muscle * (a * q2 if b.muscle_model == 0 else (q2.sqrt() / a - 1) ** 2)
        return 0.5 * b.mu * ((F * F).sum() - self.dim) - b.mu * ll + 0.5 * b.lam * ll * ll + m

    def F(self, x):
        return torch.einsum("eki,ekj->eij", x[self.T], self.S)

    def scatter(self, per_corner):
        out = torch.zeros_like(self.X)
        return out.index_add_(0, self.T.reshape(-1), per_corner.reshape(-1, self.dim))

    def energy(self, x, a):
        b = self.b
        pen = (-x[:, 1]).clamp(min=0.0)
        psi = torch.func.vmap(self.psi)(self.F(x), self.f, a)
        return (self.W * psi).sum() + (self.mass * b.gravity * x[:, 1]).sum() + b.k_contact * (pen ** 3).sum()

    def grad(self, x, a):
        """Gradient of the quasistatic energy, pinned rows dropped."""
        b = self.b
        P = torch.func.vmap(torch.func.grad(self.psi))(self.F(x), self.f, a)
        g = self.scatter(torch.einsum("e,eij,ekj->eki", self.W, P, self.S))
        g[:, 1] += self.mass * b.gravity - 3.0 * b.k_contact * (-x[:, 1]).clamp(min=0.0) ** 2
        return g * self.free[:, None]

    def potential_grad(self, x, a):
        g = self.scale * self.grad(x, a)
        if self.b.dt > 0:
            g = g + self.mass[:, None] * (x - self.hat) + self.hmask() * self.fw[:, None] * (x - self.x0)
        return g

    def hmask(self):
        return torch.tensor([1.0, 0.0, 1.0][: self.dim], dtype=torch.float64, device=DEV)

    def start(self, x0, v0):
        self.x0, self.hat = x0, x0 + self.b.dt * v0
        self.fw = 2.0 * self.b.k_friction * (self.b.eps_friction - x0[:, 1]).clamp(min=0.0)

    def linearise(self, x, a):
        d, nc = self.dim, self.dim + 1
        H = torch.func.vmap(torch.func.hessian(self.psi), chunk_size=65536)(self.F(x), self.f, a)
        self.K = torch.einsum("e,eam,eimjn,ebn->eaibj", self.scale * self.W, self.S, H, self.S).reshape(-1, nc * d, nc * d)
        self.diag = torch.zeros_like(self.X)
        self.diag[:, 1] = self.scale * 6.0 * self.b.k_contact * (-x[:, 1]).clamp(min=0.0)
        if self.b.dt > 0:
            self.diag = self.diag + self.mass[:, None] + self.hmask() * self.fw[:, None]
        self.factor = None
        n = self.X.numel()
        if n <= 6000:
            ids = (self.T[:, :, None] * d + torch.arange(d, device=DEV)).reshape(-1, nc * d)
            A = torch.zeros(n * n, dtype=torch.float64, device=DEV)
            A.index_add_(0, (ids[:, :, None] * n + ids[:, None, :]).reshape(-1), self.K.reshape(-1))
            A = A.view(n, n) + torch.diag(self.diag.reshape(-1))
            pin = (~self.free).repeat_interleave(d)
            A[pin, :], A[:, pin] = 0.0, 0.0
            A[pin, pin] = 1.0
            self.factor = torch.linalg.cholesky(A)

    def apply(self, v):
        v = v * self.free[:, None]
        y = self.scatter(torch.bmm(self.K, v[self.T].reshape(len(self.T), -1, 1)))
        return (y + self.diag * v) * self.free[:, None]

    def solve(self, rhs, rtol=1e-13):
        rhs = rhs * self.free[:, None]
        if self.factor is not None:
            x = torch.cholesky_solve(rhs.reshape(-1, 1), self.factor).view_as(rhs)
            return x + torch.cholesky_solve((rhs - self.apply(x)).reshape(-1, 1), self.factor).view_as(rhs)
        x, r, p = torch.zeros_like(rhs), rhs.clone(), rhs.clone()
        rr = (r * r).sum()
        stop = rtol * rtol * float(rr)
        for k in range(20000):
            Ap = self.apply(p)
            al = rr / (p * Ap).sum()
            x += al * p
            r -= al * Ap
            new = (r * r).sum()
            p = r + (new / rr) * p
            rr = new
            if k % 20 == 19 and float(rr) <= stop:
                break
        return x

    def minimise(self, x, a):
        g = self.potential_grad(x, a)
        g0 = float(g.norm())
        for _ in range(60):
            if float(g.norm()) <= 1e-13 * g0:
                break
            self.linearise(x, a)
            d = self.solve(-g, rtol=max(1e-13, min(1e-3, 1e-3 * float(g.norm()) / g0)))
            t = 1.0
            while t > 1e-6:
                xt = x + t * d
                gt = self.potential_grad(xt, a)
                bad = self.b.log_mode == 0 and bool((torch.linalg.det(self.F(xt)) <= 0).any())
                if not bad and float(gt.norm()) < 2.0 * float(g.norm()):
                    break
                t *= 0.5
            if float(gt.norm()) >= float(g.norm()) and float(g.norm()) <= 1e-11 * g0:
                break
            x, g = xt, gt
        return x

    def vjp(self, x, a, lam):
        """-s lam . d(grad E)/da per element."""
        q = torch.einsum("eij,ej->ei", self.F(x), self.f)
        dq = torch.einsum("eij,ej->ei", self.F(lam * self.free[:, None]), self.f)
        c, s = (q * dq).sum(dim=1), q.norm(dim=1)
        k = self.b.k_muscle
        m = k * c if self.b.muscle_model == 0 else k * (1.0 / a ** 2 - 2.0 * s / a ** 3) * c / s
        return -self.scale * self.W * m

    def material_vjp(self, x, a, lam):
        """dL/dmu, dL/dlambda, dL/dk per element (contractile muscle)."""
        F, dF = self.F(x), self.F(lam * self.free[:, None])
        J = torch.linalg.det(F)
        C = J[:, None, None] * torch.linalg.inv(F).transpose(1, 2)
        FdF, CdF = (F * dF).sum(dim=(1, 2)), (C * dF).sum(dim=(1, 2))
        ll, lp = (torch.log(J), 1.0 / J) if self.b.log_mode == 0 else ((J - 1) - 0.5 * (J - 1) ** 2, 2.0 - J)
        q, dq = torch.einsum("eij,ej->ei", F, self.f), torch.einsum("eij,ej->ei", dF, self.f)
        s = -self.scale * self.W
        return s * (FdF - lp * CdF), s * ll * lp * CdF, s * a * (q * dq).sum(dim=1)

    def step_back(self, x0, x1, v0, a, gx, gv):
        h = self.b.dt
        self.start(x0, v0)
        self.linearise(x1, a)
        lam = self.solve(gx + gv / h)
        ml = self.mass[:, None] * lam
        dx = ml - gv / h + self.hmask() * self.fw[:, None] * lam
        near = (self.fw > 0).to(lam.dtype) * 2.0 * self.b.k_friction
        dx[:, 1] += near * (self.hmask() * lam * (x1 - x0)).sum(dim=1)
        return dx, h * ml, self.vjp(x1, a, lam), lam


def exact(case, seed):
    kind, (nv, ne) = case["kind"], sizes(case)
    if (kind == "batch" and case["bodies"] > 4) or (kind == "rollout" and nv > 3000):
        return None
    if kind == "adjoint" and ne > 500e3 or kind == "quasi" and ne > 450e3 or ne > 4e6:
        return None
    v = inputs(case, seed)
    t = {k: dev(x) for k, x in v.items() if isinstance(x, np.ndarray)}
    if kind == "batch":
        return exact_batch(v, t, case["steps"])
    m = Exact(v["bodies"][0])
    if kind == "hvp":
        m.K = None
        u = t["v"].to(torch.float32).double() if case["precision"] == "mixed" else t["v"]
        F, dF = m.F(t["x"]), m.F(u * m.free[:, None])
        dP = torch.func.vmap(lambda A, B, f, a: torch.func.jvp(lambda Z: torch.func.grad(m.psi)(Z, f, a), (A,), (B,))[1],
                             chunk_size=262144)(F, dF, m.f, t["a"])
        return {"Hv": m.scatter(torch.einsum("e,eij,ekj->eki", m.W, dP, m.S)) * m.free[:, None]}
    if kind == "energy":
        return {"E": m.energy(t["x"], t["a"]), "g": m.grad(t["x"], t["a"])}
    if kind == "adjoint":
        m.linearise(t["x"], t["a"])
        lam = m.solve(t["g"])
        dmu, dlam, dk = m.material_vjp(t["x"], t["a"], lam)
        return {"lam": lam, "da": m.vjp(t["x"], t["a"], lam), "dmu": dmu, "dlam": dlam, "dk": dk}
    if kind == "quasi":
        x = m.minimise(m.X, t["a"])
        m.linearise(x, t["a"])
        lam = m.solve(((x.mean(dim=0) - t["target"]) / len(x)).expand_as(x))
        return {"x": x, "da": m.vjp(x, t["a"], lam)}
    a = t["a"] if kind == "rollout" else t["a"][None]
    x, v1, da, dx, dv, _ = exact_rollout(m, t["x0"], t["v0"], a, t["gx"], t["gv"])
    return {"x": x[-1], "v": v1[-1], "dx0": dx, "dv0": dv, "da": da if kind == "rollout" else da[0]}


def exact_rollout(m, x0, v0, a, gx, gv):
    x, v = [x0], [v0]
    for at in a:
        m.start(x[-1], v[-1])
        x.append(m.minimise(x[-1], at))
        v.append((x[-1] - x[-2]) / m.b.dt)
    da, mat = [], torch.zeros(3, dtype=torch.float64, device=DEV)
    for k in range(len(a) - 1, -1, -1):
        gx, gv, d, lam = m.step_back(x[k], x[k + 1], v[k], a[k], gx, gv)
        da.insert(0, d)
        mat += torch.stack([q.sum() for q in m.material_vjp(x[k + 1], a[k], lam)])
    return torch.stack(x), torch.stack(v), torch.stack(da), gx, gv, mat


def exact_batch(v, t, steps):
    outs, vo, eo = [], 0, 0
    for b in v["bodies"]:
        vs, es = slice(vo, vo + len(b.X)), slice(eo, eo + len(b.T))
        vo, eo = vs.stop, es.stop
        outs.append(exact_rollout(Exact(b), t["x0"][vs], t["v0"][vs], t["a"][:, es], t["gx"][vs], t["gv"][vs]))
    cat = lambda k, dim: torch.cat([o[k] for o in outs], dim=dim)  # noqa: E731
    return {"x": cat(0, 1), "v": cat(1, 1), "da": cat(2, 1), "dx0": cat(3, 0), "dv0": cat(4, 0),
            "dmat": torch.stack([o[5] for o in outs])}
