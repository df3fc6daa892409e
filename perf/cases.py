"""The work that users of the framework have it do, as cases that can be timed and compared.

A case is one kind of call on one kind of mesh:

  march         n RK4 steps of a field, then phi and psi (a simulation between two snapshots)
  precondition  psi reset from phi and relaxed in pseudo time (every 1000 steps of a simulation)
  output        the mass integrals and both fields of a large field (a monitoring or snapshot point)
  ensemble      independent instances of orders 2 to 5, one batch field per order on its own stream
  adjoint       a recorded window of RK4 steps and the gradient of a misfit at its end

Meshes are made here (grids, jittered, shuffled and rotated, squares split into triangles), inputs
from the seed (interface, velocity).  FP64 fields return FP64 values.  The mixed path's arithmetic is
single precision, and a snapshot of it is kept in single precision, so its fields come as float32.

exact() is a plain FP64 flux-reconstruction solver in torch (dense or per-axis operators, faces paired
by their centroids) of the same scheme: the march, the preconditioning and, by autograd, the adjoint.
"""
import functools
import math
import types

import numpy as np
import torch

import paper_2006_10967_gb300 as fr

GAMMA, TAU, S0, KAPPA, DELTA, PSEUDO_ITERS = 0.09, 0.1, -5.0, 5.0, 1e-12, 20


# ---------------------------------------------------------------- cases
def listed():
    return [
        # the smallest call: a translated disk on 16 x 16 quads, as in a unit test or a convergence study
        dict(name="quad16_p3_fp64", kind="march", etype="quad", nx=16, ny=16, order=3, precision="fp64",
             velocity="uniform", jitter=0.0, walls=False, steps=1),
        # the 2D benchmark: the vortex test on jittered, shuffled and rotated quads between walls
        dict(name="quad128_p4_mixed", kind="march", etype="quad", nx=128, ny=128, order=4, precision="mixed",
             velocity="rider_kothe", jitter=0.1, walls=True, steps=16),
        # an ordinary 2D run of odd sizes at the other orders: solid-body rotation
        dict(name="quad211x187_p3_mixed", kind="march", etype="quad", nx=211, ny=187, order=3, precision="mixed",
             velocity="rotation", jitter=0.0, walls=False, steps=8),
        # the triangle benchmark: about 30,000 triangles of order 3
        dict(name="tri122_p3_mixed", kind="march", etype="tri", nx=122, ny=122, order=3, precision="mixed",
             velocity="rider_kothe", jitter=0.1, walls=True, steps=8),
        # the 3D benchmark and the largest call: the LeVeque deformation on 64^3 hexes
        dict(name="hex64_p3_mixed", kind="march", etype="hex", nx=64, ny=64, nz=64, order=3, precision="mixed",
             velocity="leveque", jitter=0.0, walls=True, steps=2),
        # the same flow at the next order of the paper's sweep
        dict(name="hex32_p4_mixed", kind="march", etype="hex", nx=32, ny=32, nz=32, order=4, precision="mixed",
             velocity="leveque", jitter=0.0, walls=True, steps=2),
        # an unstructured hex mesh: jittered, shuffled, rotated elements of ragged counts
        dict(name="hex27x22x19_p2_mixed", kind="march", etype="hex", nx=27, ny=22, nz=19, order=2,
             precision="mixed", velocity="uniform", jitter=0.1, walls=False, steps=4),
        # the plain FP64 path that accuracy studies use
        dict(name="hex24_p3_fp64", kind="march", etype="hex", nx=24, ny=24, nz=24, order=3, precision="fp64",
             velocity="leveque", jitter=0.0, walls=True, steps=1),
        # the preconditioning of a 3D run
        dict(name="precondition_hex40_p3_mixed", kind="precondition", etype="hex", nx=40, ny=40, nz=40, order=3,
             precision="mixed", velocity="leveque", jitter=0.0, walls=True),
        # what a 3D run writes out and monitors
        dict(name="output_hex48_p3_mixed", kind="output", etype="hex", nx=48, ny=48, nz=48, order=3,
             precision="mixed", velocity="leveque", jitter=0.0, walls=True),
        # the batched ensemble: uneven periodic instances with velocities of their own
        dict(name="ensemble24_mixed", kind="ensemble", instances=24, nmin=16, nmax=96, precision="mixed", steps=8),
        # the inverse problem: gradient of a final misfit with respect to the fields and the velocity
        dict(name="adjoint_quad64_p4_fp64", kind="adjoint", etype="quad", nx=64, ny=64, order=4, precision="fp64",
             velocity="stream", jitter=0.0, walls=False, steps=20, ckpt=10),
    ]


def _sizes(rng, lo, hi, axes):
    """Grid counts of about one size, drawn evenly over its logarithm, each axis of its own."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return {a: min(int(hi), max(lo, int(round(n * rng.uniform(0.75, 1.3))))) for a in axes}


def draw(rng):
    kind = rng.choice(["march"] * 7 + ["precondition"] * 2 + ["output", "ensemble", "adjoint"])
    if kind == "ensemble":
        nmax = rng.randint(32, 96)
        return dict(kind=kind, instances=rng.randint(5, 24), nmin=rng.randint(8, 24), nmax=nmax, precision="mixed",
                    steps=rng.randint(2, 8))
    if kind == "adjoint":
        n, p = rng.randint(12, 56), rng.randint(2, 4)
        return dict(kind=kind, etype="quad", nx=n, ny=rng.randint(12, 56), order=p, precision="fp64",
                    velocity="stream", jitter=0.0, walls=False, steps=10 * rng.randint(1, 2), ckpt=5)
    etype = rng.choice(["quad", "quad", "tri", "hex", "hex", "hex"])
    mixed = rng.random() < 0.8
    c = dict(kind=kind, etype=etype, precision="mixed" if mixed else "fp64")
    if etype == "hex":
        c["order"] = rng.choice([1, 2, 3, 3, 3, 4, 5])
        top = (64 if mixed else 24) * 4 / (c["order"] + 1)
        if kind == "precondition":
            top *= 0.6
        c.update(_sizes(rng, 6, max(8, top), ("nx", "ny", "nz")))
        c["velocity"] = rng.choice(["leveque", "leveque", "uniform"])
    else:
        c["order"] = rng.randint(1, 6 if etype == "quad" else 4)
        top = (400 if mixed else 120) * (1.0 if etype == "quad" else 0.6)
        if kind == "precondition":
            top *= 0.5
        c.update(_sizes(rng, 8, top, ("nx", "ny")))
        c["velocity"] = rng.choice(["rider_kothe", "uniform", "rotation", "stream"])
    c["walls"] = c["velocity"] in ("rider_kothe", "leveque") and rng.random() < 0.6
    c["jitter"] = rng.choice([0.0, 0.1])
    if kind == "march":
        pts = _counts(etype, c["order"])[0] * c["nx"] * c["ny"] * c.get("nz", 1) * (2 if etype == "tri" else 1)
        c["steps"] = min(rng.randint(1, 4), 1 + int((3e7 if mixed else 1.5e6) / pts))
    return c


# ---------------------------------------------------------------- meshes
class Grid(types.SimpleNamespace):
    """etype, nodes, conn, periodic, period: what fr.Mesh takes."""


@functools.lru_cache(maxsize=None)
def _grid(etype, ns, jitter, walls, length):
    """A grid of quads, of squares split into triangles, or of hexes on [0, length]^dim.  With jitter the inner
    nodes are moved by up to that share of the spacing (images of a periodic node alike), the elements are
    shuffled and their vertex lists rotated."""
    dim = len(ns)
    rng = np.random.default_rng(7)
    nodes = np.stack([m.ravel(order="F") for m in
                      np.meshgrid(*[np.linspace(0.0, length, n + 1) for n in ns], indexing="ij")], 1)
    if jitter:
        idx = np.stack(np.unravel_index(np.arange(len(nodes)), [n + 1 for n in ns], order="F"), 1)
        key = idx if walls else idx % np.array(ns)
        move = rng.uniform(-jitter, jitter, (len(nodes), dim)) * (length / np.array(ns))
        move = move[np.ravel_multi_index(key.T, [n + 1 for n in ns], order="F")]
        if walls:
            move[(idx == 0) | (idx == np.array(ns))] = 0.0
        nodes = nodes + move
    at = np.stack([m.ravel(order="F") for m in np.meshgrid(*[np.arange(n) for n in ns], indexing="ij")])
    corner = [(0, 0), (1, 0), (1, 1), (0, 1)]
    corner = corner if dim == 2 else [c + (z,) for z in (0, 1) for c in corner]
    step = np.cumprod([1] + [n + 1 for n in ns[:-1]])
    conn = np.stack([((at + np.array(c)[:, None]) * step[:, None]).sum(0) for c in corner], 1)
    if etype == "tri":
        conn = np.concatenate([conn[:, [0, 1, 2]], conn[:, [0, 2, 3]]], 0)
    if jitter:
        conn = conn[rng.permutation(len(conn))]
        turns = [[0, 1, 2], [1, 2, 0], [2, 0, 1]] if etype == "tri" else [[(k + r) % 4 for k in range(4)] for r in range(4)]
        if dim == 3:  # quarter turns about the third axis, and the half turn about the first
            quarter = [[t[k % 4] + 4 * (k // 4) for k in range(8)] for t in turns]
            turns = quarter + [[t[7 - k] for k in range(8)] for t in quarter]
        conn = np.take_along_axis(conn, np.array(turns)[rng.integers(0, len(turns), len(conn))], 1)
    return Grid(etype=etype, nodes=nodes, conn=conn.astype(np.int64), periodic=(not walls,) * dim, period=(length,) * dim)


def _grid_of(case):
    ns = tuple(case[a] for a in ("nx", "ny", "nz") if a in case)
    return _grid(case["etype"], ns, case["jitter"], case["walls"], 4.0 if case["velocity"] == "rotation" else 1.0)


@functools.lru_cache(maxsize=None)
def _mesh(etype, ns, jitter, walls, length, order):
    """A program builds its host mesh once and makes its fields on it."""
    return fr.Mesh.from_synthetic(_grid(etype, ns, jitter, walls, length), order)


def _mesh_of(case):
    ns = tuple(case[a] for a in ("nx", "ny", "nz") if a in case)
    return _mesh(case["etype"], ns, case["jitter"], case["walls"], 4.0 if case["velocity"] == "rotation" else 1.0,
                 case["order"])


# ---------------------------------------------------------------- problems
def _stream(rng, modes=16):
    """A random-phase stream function, |k| <= 4, spectrum 1/|k|^2, largest speed 1."""
    pool = [(kx, ky) for kx in range(5) for ky in range(-4, 5) if (kx or ky > 0) and kx * kx + ky * ky <= 16]
    k = np.array([pool[i] for i in rng.choice(len(pool), modes, replace=False)], dtype=np.float64)
    th = rng.uniform(0, 2 * np.pi, modes)
    a = 1.0 / (k ** 2).sum(1)
    v = types.SimpleNamespace(kind="stream", a=(0.0, 0.0, 0.0), T=4.0, kx=k[:, 0].copy(), ky=k[:, 1].copy(),
                              A=a * np.cos(th), B=a * np.sin(th))
    g = torch.stack(torch.meshgrid(*[torch.linspace(0, 1, 129, dtype=torch.float64)] * 2, indexing="ij"), -1)
    top = float(_velocity(v, g).norm(dim=-1).max())
    v.A, v.B = v.A / top, v.B / top
    return v


def _problem(velocity, etype, dim, order, h, rng):
    """The record that fr.make_params takes, and the initial interface, with the paper's parameters."""
    length, vmax, T, a = 1.0, 1.0, 0.0, (0.0, 0.0, 0.0)
    if velocity == "uniform":
        a = tuple(rng.uniform(0.4, 1.0, 3)[:dim]) + (0.0,) * (3 - dim)
        vmax = math.sqrt(sum(x * x for x in a))
    elif velocity == "rider_kothe":
        T = 8.0
    elif velocity == "leveque":
        T, vmax = 3.0, 2.0
    elif velocity == "rotation":
        length, a = 4.0, (2.0, 2.0, 0.0)
        vmax = math.sqrt(8.0)
    v = _stream(rng) if velocity == "stream" else types.SimpleNamespace(kind=velocity, a=a, T=T)
    r = length * rng.uniform(0.13, 0.2)
    centre = tuple(length * rng.uniform(0.35, 0.65, dim))
    circle = types.SimpleNamespace(centre=centre, radius=r, beta=3 * order / (4 * h))
    w = types.SimpleNamespace(
        gamma=GAMMA, eps=0.06 * h / order, tau=TAU, tau_psi=TAU, tau_pseudo=TAU, dt=0.1 * h / ((order + 1) * vmax),
        n_precond=1000, pseudo_kmax=PSEUDO_ITERS, pseudo_dtau=0.1 * h / (order + 1), pseudo_tol=0.5, s0=S0,
        kappa=KAPPA, nu_max=0.15 * h / order, delta=DELTA, velocity=v, circle=circle, order=order)
    return w


def _problem_of(case, seed, h):
    dim = 3 if case["etype"] == "hex" else 2
    w = _problem(case["velocity"], case["etype"], dim, case["order"], h, np.random.default_rng(seed))
    if case["kind"] == "adjoint":
        w.n_precond = 1 << 30  # a recorded window holds no preconditioning
        w.velocity.T = 0.0
    return w


def _instances(case, seed):
    """The ensemble: uneven grids (the same for every seed), velocities and disks from the seed."""
    size = np.random.default_rng(case["instances"])
    rng = np.random.default_rng(seed)
    out = []
    for i in range(case["instances"]):
        n = int(size.integers(case["nmin"], case["nmax"] + 1))
        w = _problem("stream", "quad", 2, 2 + i % 4, 1.0 / n, rng)
        w.n = n
        w.mesh = functools.partial(_grid, "quad", (n, n), 0.0, False, 1.0)
        out.append(w)
    return out


def prepare(case, seed):
    if case["kind"] == "ensemble":
        groups = fr.batch_from_workloads(_instances(case, seed), case["precision"], pseudo_fixed=True)
        return types.SimpleNamespace(case=case, groups=groups, streams=[torch.cuda.Stream() for _ in groups])
    m = _mesh_of(case)
    w = _problem_of(case, seed, m.info.h)
    f = fr.Field(m, fr.make_params(w, case["precision"], pseudo_fixed=True), ic=w.circle, precondition=True)
    s = types.SimpleNamespace(case=case, field=f, shape=m.shape)
    if case["kind"] == "adjoint":
        x = torch.from_numpy(m.solution_points()).cuda()
        s.weights = torch.from_numpy(m.quadrature()).cuda()
        s.target = _target(x, w)
        s.n_coef = 2 * len(w.velocity.A)
    return s


def _target(x, w):
    """The interface that the adjoint's misfit compares with: the disk, moved and grown."""
    c = w.circle
    d = (x - torch.tensor(c.centre, dtype=torch.float64, device=x.device) - 0.05).norm(dim=-1)
    return 0.5 * (1 + torch.tanh(c.beta * (1.1 * c.radius - d)))


def _snapshot(field, case):
    keep = torch.float64 if case["precision"] == "fp64" else torch.float32
    shape = field.mesh.shape
    return [field.get_device(i, torch.empty(shape, dtype=torch.float64, device="cuda")).to(keep) for i in (0, 1)]


def run(state):
    case = state.case
    if case["kind"] == "ensemble":
        here = torch.cuda.current_stream()
        for (_, f, _), s in zip(state.groups, state.streams):
            s.wait_stream(here)
            f.step(case["steps"], stream=s)
        for s in state.streams:
            here.wait_stream(s)
        return [_snapshot(f, case) for _, f, _ in state.groups]
    f = state.field
    if case["kind"] == "march":
        f.step(case["steps"])
        return _snapshot(f, case)
    if case["kind"] == "precondition":
        f.precondition()
        return _snapshot(f, case)[1]
    if case["kind"] == "output":
        return [f.mass(0), f.mass(1)] + _snapshot(f, case)
    f.adjoint_record(case["steps"], case["ckpt"])
    phi = f.get_device(0, torch.empty(state.shape, dtype=torch.float64, device="cuda"))
    du0, dcoef = f.adjoint_step(state.weights * (phi - state.target), None, state.n_coef)
    return [phi, du0, dcoef]


# ---------------------------------------------------------------- what a pass cannot do without
def _counts(etype, order):
    """Solution points, flux points and floating operations of one residual of one field per element: the
    operator applies of Steps 1, 3, 5 and 6 (per axis on quads and hexes, dense on triangles) and 30 a point."""
    n = order + 1
    if etype == "tri":
        nu, nf = n * (n + 1) // 2, 3 * n
        return nu, nf, 2 * (nf * nu * 4 + nu * nu * 4 + nu * nf * 2) + 30 * nu
    dim = 2 if etype == "quad" else 3
    nu, nf = n ** dim, 2 * dim * n ** (dim - 1)
    return nu, nf, 2 * dim * nu * (2 * n + 8) + 30 * nu + 30 * nf


def work(case):
    b = 8 if case["precision"] == "fp64" else 4
    keep = b
    if case["kind"] == "ensemble":
        size, tot = np.random.default_rng(case["instances"]), dict(bytes=0, flops=0)
        for i in range(case["instances"]):
            n = int(size.integers(case["nmin"], case["nmax"] + 1))
            one = work(dict(kind="march", etype="quad", nx=n, ny=n, order=2 + i % 4, precision="mixed", steps=case["steps"]))
            tot = {k: tot[k] + one[k] for k in tot}
        return tot
    nu, nf, ops = _counts(case["etype"], case["order"])
    E = case["nx"] * case["ny"] * case.get("nz", 1) * (2 if case["etype"] == "tri" else 1)
    pts = E * nu
    # a stage: the stage value read and written, the solution (FP64 or a pair) read, the accumulator read and
    # written, for both fields; traces and common fluxes of half the face points each written and read
    stage = pts * 2 * (2 * b + 8 + 2 * b) + E * nf * 2 * (2 * b)
    pseudo = pts * (2 * b + 8 + 2 * b + 8) + E * nf * (2 * b)
    if case["kind"] == "march":
        return dict(bytes=4 * case["steps"] * stage + 2 * pts * keep, flops=4 * case["steps"] * 2 * E * ops)
    if case["kind"] == "precondition":
        return dict(bytes=4 * PSEUDO_ITERS * pseudo + pts * keep, flops=4 * PSEUDO_ITERS * E * ops)
    if case["kind"] == "output":
        return dict(bytes=pts * (2 * 8 + 8) + 2 * pts * keep, flops=8 * pts)
    n = 4 * case["steps"]  # forward, recomputation and the reverse of every stage
    return dict(bytes=n * 4 * stage, flops=n * 4 * 2 * E * ops)


# ---------------------------------------------------------------- the same scheme in plain FP64 torch
def _velocity(v, x, coef=None):
    """The spatial factor of the velocity at points x (..., dim)."""
    pi, X, Y = math.pi, x[..., 0], x[..., 1]
    s2 = lambda t: torch.sin(pi * t) ** 2  # noqa: E731
    d2 = lambda t: torch.sin(2 * pi * t)  # noqa: E731
    if v.kind == "uniform":
        return torch.tensor(v.a[: x.shape[-1]], dtype=torch.float64, device=x.device).expand(x.shape)
    if v.kind == "rider_kothe":
        return torch.stack([-s2(X) * d2(Y), d2(X) * s2(Y)], -1)
    if v.kind == "leveque":
        Z = x[..., 2]
        return torch.stack([2 * s2(X) * d2(Y) * d2(Z), -d2(X) * s2(Y) * d2(Z), -d2(X) * d2(Y) * s2(Z)], -1)
    if v.kind == "rotation":
        return torch.stack([v.a[1] - Y, X - v.a[0]], -1)
    t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=x.device)  # noqa: E731
    A, B = (t(v.A), t(v.B)) if coef is None else (coef[: len(v.A)], coef[len(v.A):])
    kx, ky = t(v.kx), t(v.ky)
    arg = 2 * pi * (X[..., None] * kx + Y[..., None] * ky)
    d = 2 * pi * (A * torch.cos(arg) - B * torch.sin(arg))
    return torch.stack([(d * ky).sum(-1), -(d * kx).sum(-1)], -1)


def _legendre(x, m):
    return np.polynomial.legendre.legval(x, [0] * m + [math.sqrt(m + 0.5)])


class _Line:
    """1D operators of n Gauss-Legendre points: derivative, end interpolation, Radau lifts, orthonormal modes."""

    def __init__(self, n, dev):
        x, w = np.polynomial.legendre.leggauss(n)
        V = np.stack([_legendre(x, m) for m in range(n)], 1)
        dV = np.stack([np.polynomial.legendre.legval(x, np.polynomial.legendre.legder([0] * m + [math.sqrt(m + 0.5)]))
                       for m in range(n)], 1)
        Vi = np.linalg.inv(V)
        end = [np.array([_legendre(s, m) for m in range(n)]) @ Vi for s in (-1.0, 1.0)]
        t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.x, self.w, self.D, self.end, self.modes = x, w, t(dV @ Vi), t(np.stack(end)), t(Vi)
        self.lift = t(np.stack([end[0] / w, end[1] / w]))  # of the outward flux at the left and the right end


class _Tensor:
    """Quads and hexes: values (E, fields, nu), axis a of the points reached through a view."""

    def __init__(self, dim, n, dev):
        self.dim, self.n, self.o = dim, n, _Line(n, dev)
        self.nu, self.nfp, self.nfaces = n ** dim, n ** (dim - 1), 2 * dim
        self.nf = self.nfaces * self.nfp
        x = self.o.x
        pts = np.stack([np.tile(np.repeat(x, n ** b), n ** (dim - 1 - b)) for b in range(dim)], 1)
        face = []
        for a in range(dim):
            for s in (-1.0, 1.0):
                q = [np.tile(np.repeat(x, n ** b), n ** (dim - 2 - b)) for b in range(dim - 1)]
                q.insert(a, np.full(self.nfp, s))
                face.append(np.stack(q, 1))
        self.xu, self.xf = pts, np.concatenate(face)
        self.nref = np.repeat(np.concatenate([[-np.eye(dim)[a], np.eye(dim)[a]] for a in range(dim)]), self.nfp, 0)
        self.wq = functools.reduce(np.multiply, [np.tile(np.repeat(self.o.w, n ** b), n ** (dim - 1 - b)) for b in range(dim)])
        top = functools.reduce(np.logical_or, [np.tile(np.repeat(np.arange(n), n ** b), n ** (dim - 1 - b)) == n - 1 for b in range(dim)])
        self.top = torch.tensor(top, device=dev)
        l = np.arange(self.nfp)
        self.orders = [l, l[::-1].copy()]
        if dim == 3:
            i, j = l % n, l // n
            self.orders = [(n - 1 - a if r & 1 else a) + n * (n - 1 - b if r & 2 else b)
                           for a, b in ((i, j), (j, i)) for r in range(4)]
        r = lambda *c: np.array(c, dtype=np.float64)  # noqa: E731
        c2 = [r(-1, -1), r(1, -1), r(1, 1), r(-1, 1)]
        self.corners = np.array(c2 if dim == 2 else [np.append(c, z) for z in (-1.0, 1.0) for c in c2])

    def shape(self, xi):  # vertex weights and their reference gradients at points xi
        f = 0.5 * (1 + self.corners[None] * xi[:, None])
        N = f.prod(-1)
        G = np.stack([0.5 * self.corners[None, :, a] * np.delete(f, a, -1).prod(-1) for a in range(self.dim)], -1)
        return N, G

    def _along(self, M, U, a):
        n, d = self.n, self.dim
        V = U.reshape(-1, n ** (d - 1 - a), n, n ** a)
        return torch.einsum("ij,bpjq->bpiq", M, V)

    def trace(self, U):
        return torch.cat([self._along(self.o.end, U, a).transpose(1, 2).reshape(U.shape[:-1] + (2 * self.nfp,))
                          for a in range(self.dim)], -1)

    def deriv(self, U, a):
        return self._along(self.o.D, U, a).reshape(U.shape)

    def lift(self, c, a=None):
        """Lift of outward normal values c at the flux points (of axis a's faces, or all)."""
        n, d, out = self.n, self.dim, 0
        for b in range(d) if a is None else (a,):
            k = c[..., 2 * b * self.nfp:2 * (b + 1) * self.nfp].reshape(-1, 2, n ** (d - 1 - b), n ** b)
            out = out + torch.einsum("sj,bspq->bpjq", self.o.lift, k).reshape(c.shape[:-1] + (self.nu,))
        return out

    def modes(self, U):
        for a in range(self.dim):
            U = self._along(self.o.modes, U, a).reshape(U.shape)
        return U


class _Triangle:
    """Triangles: dense operators from the monomial basis, on the Blyth-Pozrikidis points."""
    dim, nfaces = 2, 3

    def __init__(self, n, dev):
        g, w = np.polynomial.legendre.leggauss(n)
        p = n - 1
        v = 0.5 * (g + 1) if p != 5 else 0.5 * (np.cos((n - np.arange(n)) * np.pi / (n + 1)) + 1)
        pts = []
        for j in range(n):
            for i in range(n - j):
                a, b, c = v[i], v[j], v[p - i - j]
                l1, l2 = (1 + 2 * a - b - c) / 3, (1 + 2 * b - a - c) / 3
                pts.append((2 * l1 - 1, 2 * l2 - 1))
        self.corners = np.array([(-1.0, -1.0), (1.0, -1.0), (-1.0, 1.0)])
        lam = 0.5 * (1 + g)[:, None]
        self.xu = np.array(pts)
        self.xf = np.concatenate([(1 - lam) * self.corners[e] + lam * self.corners[(e + 1) % 3] for e in range(3)])
        r = math.sqrt(0.5)
        self.nref = np.repeat(np.array([(0, -1), (r, r), (-1.0, 0)]), n, 0)
        wf = np.concatenate([w * 0.5 * L for L in (2.0, 2.0 / r, 2.0)])
        self.nu, self.nfp, self.nf = len(pts), n, 3 * n
        self.orders = [np.arange(n), np.arange(n)[::-1].copy()]
        ex = [(i, k - i) for k in range(n) for i in range(k + 1)]
        basis = lambda x: np.stack([x[:, 0] ** i * x[:, 1] ** j for i, j in ex], 1)  # noqa: E731
        dr = lambda x: np.stack([i * x[:, 0] ** max(i - 1, 0) * x[:, 1] ** j for i, j in ex], 1)  # noqa: E731
        ds = lambda x: np.stack([j * x[:, 0] ** i * x[:, 1] ** max(j - 1, 0) for i, j in ex], 1)  # noqa: E731
        # Gram matrix by collapsed Gauss quadrature; degrees ascend, so its Cholesky factor gives orthonormal modes
        q, wq = np.polynomial.legendre.leggauss(n + 2)
        A, B = np.meshgrid(q, q, indexing="ij")
        xq = np.stack([((1 + A) * (1 - B) / 2 - 1).ravel(), B.ravel()], 1)
        ww = (np.outer(wq, wq) * (1 - B) / 2).ravel()
        Bq = basis(xq)
        C = np.linalg.cholesky(Bq.T @ (ww[:, None] * Bq))  # modes = monomials C^-T
        Ci = np.linalg.inv(C).T
        V = basis(self.xu) @ Ci
        Vi = np.linalg.inv(V)
        L = basis(self.xf) @ Ci @ Vi
        t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.L, self.D, self.V = t(L), [t(f(self.xu) @ Ci @ Vi) for f in (dr, ds)], t(Vi)
        self.LIFT = t((V @ V.T) @ (L.T * wf))
        self.n_ = t(self.nref)
        self.wq = (Bq @ Ci @ Vi).T @ ww
        self.top = torch.tensor([i + j == p for i, j in ex], device=dev)

    def shape(self, xi):
        N = np.stack([-(xi[:, 0] + xi[:, 1]) / 2, (1 + xi[:, 0]) / 2, (1 + xi[:, 1]) / 2], 1)
        G = np.broadcast_to(np.array([(-0.5, -0.5), (0.5, 0), (0, 0.5)]), (len(xi), 3, 2))
        return N, G

    def trace(self, U):
        return U @ self.L.T

    def deriv(self, U, a):
        return U @ self.D[a].T

    def lift(self, c, a=None):
        return (c if a is None else c * self.n_[:, a].abs()) @ self.LIFT.T

    def modes(self, U):
        return U @ self.V.T


class _Scheme:
    """Geometry, face pairing and the residuals of one mesh."""

    def __init__(self, grid, order, dev):
        n, dim = order + 1, grid.nodes.shape[1]
        self.el = el = _Triangle(n, dev) if grid.etype == "tri" else _Tensor(dim, n, dev)
        self.dim, self.dev, self.tri = dim, dev, grid.etype == "tri"
        t = lambda a: torch.tensor(np.ascontiguousarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        X = t(grid.nodes)[torch.as_tensor(grid.conn, device=dev)]  # E, verts, dim
        (Nu, Gu), (Nf, Gf) = el.shape(el.xu), el.shape(el.xf)
        self.x, self.xf = torch.einsum("iv,evc->eic", t(Nu), X), torch.einsum("kv,evc->ekc", t(Nf), X)
        # adjugates S = det J J^-1 at the solution points, and the transformed normals det J J^-T n~ at the flux points
        J = torch.einsum("iva,evc->eica", t(Gu), X)
        self.det, self.S = self._adjugate(J)
        self.wdet = t(el.wq) * self.det
        Sf = self._adjugate(torch.einsum("kva,evc->ekca", t(Gf), X))[1]
        pn = torch.einsum("ekac,ka->ekc", Sf, t(el.nref))
        self.pm = pn.norm(dim=-1)
        self.nh = pn / self.pm[..., None]
        E = X.shape[0]
        self.h = float((2 * self.wdet.sum() / E) ** 0.5 if self.tri else (self.wdet.sum() / E) ** (1 / dim))
        self._pair(grid, X)

    @staticmethod
    def _adjugate(J):
        if J.shape[-1] == 2:
            a, b, c, d = J[..., 0, 0], J[..., 0, 1], J[..., 1, 0], J[..., 1, 1]
            return a * d - b * c, torch.stack([torch.stack([d, -b], -1), torch.stack([-c, a], -1)], -2)
        r = [J[..., k] for k in range(3)]  # columns; the adjugate's rows are their cross products
        S = torch.stack([torch.linalg.cross(r[1], r[2]), torch.linalg.cross(r[2], r[0]), torch.linalg.cross(r[0], r[1])], -2)
        return (r[0] * S[..., 0, :]).sum(-1), S

    def _pair(self, grid, X):
        """Partner flux point of every flux point (its own at a wall), and whether it is an L point: the element
        of the lower number has the L side."""
        el, dev = self.el, self.dev
        E, F = X.shape[0], el.nfaces
        P = self.xf.reshape(E, F, el.nfp, self.dim)
        per = torch.tensor(grid.period, dtype=torch.float64, device=dev)
        wrap = grid.periodic[0]
        q = 2.0 ** 20
        key = torch.floor(P.mean(2) / per * q + 0.3137).long()
        if wrap:
            key = key % int(q)
        key = functools.reduce(lambda a, b: a * (1 << 21) + b, [key[..., a] for a in range(self.dim)]).reshape(-1)
        key, at = torch.sort(key, stable=True)
        same = torch.nonzero(key[1:] == key[:-1]).reshape(-1)
        one, two = at[same], at[same + 1]
        me = torch.arange(E * el.nf, device=dev).reshape(E * F, el.nfp)
        other, is_l = me.clone(), torch.ones(E * F, dtype=torch.bool, device=dev)
        Pf = P.reshape(E * F, el.nfp, self.dim)
        best, far = None, None
        for o in el.orders:
            o = torch.as_tensor(o, device=dev)
            d = Pf[one] - Pf[two][:, o]
            if wrap:
                d = d - per * torch.round(d / per)
            d = d.abs().amax((1, 2))
            pick = me[two][:, o]
            best = pick if best is None else torch.where((d < far)[:, None], pick, best)
            far = d if far is None else torch.minimum(d, far)
        assert far.numel() == 0 or float(far.max()) < 1e-6 * self.h
        other[one] = best
        other.view(-1)[best.reshape(-1)] = me[one].reshape(-1)
        first = one // F < two // F
        is_l[one], is_l[two] = first, ~first
        self.other, self.isl = other.reshape(E, el.nf), is_l[:, None].expand(-1, el.nfp).reshape(E, el.nf)

    def partner(self, f):  # f: E, fields, nf
        flat = f.transpose(1, 2).reshape(-1, f.shape[1])
        return flat[self.other].transpose(1, 2)

    def gradient(self, U, uf, uo):
        jump = torch.where(self.isl[:, None], uo - uf, torch.zeros_like(uf))
        q = []
        n = torch.tensor(self.el.nref, dtype=torch.float64, device=self.dev)
        for a in range(self.dim):
            lifted = self.el.lift(jump * n[:, a]) if self.tri else self.el.lift(jump * n[:, a], a)
            q.append(self.el.deriv(U, a) + lifted)
        return [sum(self.S[:, None, :, a, c] * q[a] for a in range(self.dim)) / self.det[:, None] for c in range(self.dim)]

    def divergence(self, f, F):
        """F: the common normal flux out of the L side (physical on triangles, transformed elsewhere)."""
        Fo = torch.where(self.isl[:, None], F, -self.partner(F))
        if self.tri:
            Fo = Fo * self.pm[:, None]
        n = torch.tensor(self.el.nref, dtype=torch.float64, device=self.dev)
        out = 0
        for a in range(self.dim):
            fa = sum(self.S[:, None, :, a, c] * f[c] for c in range(self.dim))
            out = out + self.el.deriv(fa, a)
            Fo = Fo - n[:, a] * self.el.trace(fa)
        return out + self.el.lift(Fo)

    def rate(self, U, w, g, coef=None):
        """dU/dt of U = [phi, psi] (E, 2, nu), time factor g."""
        if coef is not None or not hasattr(self, "v"):
            v, vf = _velocity(w.velocity, self.x, coef), _velocity(w.velocity, self.xf, coef)
            if coef is None:
                self.v, self.vf = v, vf
        else:
            v, vf = self.v, self.vf
        v, vf = g * v, g * vf
        uf = self.el.trace(U)
        uo = self.partner(uf)
        q = self.gradient(U, uf, uo)
        qf = [self.el.trace(c) for c in q]

        def viscous(u, qs, vel):
            M = vel.norm(dim=-1).clamp(min=w.gamma)
            gm = torch.sqrt(sum(c[:, 1] ** 2 for c in qs).clamp(min=w.delta ** 2))
            return [M * (w.eps * c[:, 0] - w.gamma * u * (1 - u) * c[:, 1] / gm) for c in qs]

        vis = viscous(U[:, 0], q, v)
        f = [torch.stack([U[:, 0] * v[..., c] - vis[c], U[:, 1] * v[..., c]], 1) for c in range(self.dim)]
        visf = viscous(uf[:, 0], qf, vf)
        vn = (vf * self.nh).sum(-1)
        F = 0.5 * (uf + uo) * vn[:, None] + TAU * (uf - uo)
        F = torch.stack([F[:, 0] - sum(self.nh[..., c] * visf[c] for c in range(self.dim)), F[:, 1]], 1)
        if not self.tri:
            F = F * self.pm[:, None]
        return -self.divergence(f, F) / self.det[:, None]

    def pseudo_rate(self, psi, psi0, w):
        U = psi[:, None]
        uf = self.el.trace(U)
        uo = self.partner(uf)
        q = self.gradient(U, uf, uo)
        e = self.el.modes(U)[:, 0] ** 2
        hi, tot = (e * self.el.top).sum(-1), e.sum(-1)
        s = torch.log10(hi / tot)
        ramp = 0.5 * w.nu_max * (1 + torch.sin(math.pi * (s - w.s0) / (2 * w.kappa)))
        nu = torch.where(s < w.s0 - w.kappa, 0 * ramp, torch.where(s > w.s0 + w.kappa, 0 * ramp + w.nu_max, ramp))
        nu = torch.where((hi > 0) & (tot > 0), nu, torch.zeros_like(nu))[:, None, None]
        f = [-nu * c for c in q]
        F = TAU * (uf - uo) - nu * sum(self.nh[..., c][:, None] * self.el.trace(q[c]) for c in range(self.dim))
        if not self.tri:
            F = F * self.pm[:, None]
        qm = torch.sqrt(sum(c[:, 0] ** 2 for c in q))
        source = torch.tanh(psi0 / qm.clamp(min=w.delta)) * (1 - qm)
        return source - self.divergence(f, F)[:, 0] / self.det

    def start(self, w):
        c = w.circle
        d = (self.x - torch.tensor(c.centre, dtype=torch.float64, device=self.dev)).norm(dim=-1)
        return 0.5 * (1 + torch.tanh(c.beta * (c.radius - d)))

    def precondition(self, phi, w):
        psi0 = phi - 0.5
        return _rk4(lambda y, _: self.pseudo_rate(y, psi0, w), psi0, 0.0, w.pseudo_dtau, PSEUDO_ITERS)

    def march(self, U, w, steps, coef=None):
        T = w.velocity.T
        g = lambda t: math.cos(math.pi * t / T) if T > 0 and w.velocity.kind != "rotation" else 1.0  # noqa: E731
        return _rk4(lambda y, t: self.rate(y, w, g(t), coef), U, 0.0, w.dt, steps)


def _rk4(f, y, t, dt, steps):
    for _ in range(steps):
        a = f(y, t)
        b = f(y + 0.5 * dt * a, t + 0.5 * dt)
        c = f(y + 0.5 * dt * b, t + 0.5 * dt)
        d = f(y + dt * c, t + dt)
        y = y + dt / 6 * (a + 2 * b + 2 * c + d)
        t = t + dt
    return y


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] == "ensemble":
        out = {}
        with torch.no_grad():
            for w in _instances(case, seed):
                s = _Scheme(w.mesh(), w.order, dev)
                phi = s.start(w)
                U = s.march(torch.stack([phi, s.precondition(phi, w)], 1), w, case["steps"])
                out.setdefault(w.order, []).append(U)
        return [[torch.cat(out[p])[:, i].contiguous() for i in (0, 1)] for p in sorted(out)]
    s = _Scheme(_grid_of(case), case["order"], dev)
    w = _problem_of(case, seed, s.h)
    with torch.no_grad():
        phi = s.start(w)
        psi = s.precondition(phi, w)
        U = torch.stack([phi, psi], 1)
        if case["kind"] == "precondition":
            return psi
        if case["kind"] == "output":
            return [float((s.wdet * phi).sum()), float((s.wdet * psi).sum()), phi, psi]
        if case["kind"] == "march":
            U = s.march(U, w, case["steps"])
            return [U[:, 0].contiguous(), U[:, 1].contiguous()]
    coef = torch.tensor(np.concatenate([w.velocity.A, w.velocity.B]), dtype=torch.float64, device=dev, requires_grad=True)
    U.requires_grad_(True)
    V = s.march(U, w, case["steps"], coef)
    with torch.no_grad():
        g = s.wdet * (V[:, 0] - _target(s.x, w))
    dU, dc = torch.autograd.grad((V[:, 0] * g).sum(), (U, coef))
    return [V[:, 0].detach(), dU.transpose(0, 1).contiguous(), dc]
