"""The work that users of the library have it do, as measurable cases.

A case is one of
  * a run of a few IPCS time steps on a mesh, from fields that the program sets
    (a restart, or one member of an ensemble on the same mesh) to the fields that it
    reads back: ``what = "steps"``;
  * the network of the learned pressure guess: inference (``"guess"``) and one training
    sample's loss and gradient (``"train"``);
  * the stand-alone sparse products (``"products"``).

Meshes are triangulated boxes and channels of any size, with the vertices moved off the grid
or not, numbered lexicographically, by reverse Cuthill-McKee or at random (a mesh generator's
order).  The mesh and its multigrid hierarchy are made once and kept, as a program does;
every prepared state has a solver and fields of its own.

The solves end at the relative residuals of the repository's own runs: 1e-8 in mixed precision,
1e-12 in float64.  A mixed run is good to about seven digits (its matrix and its velocity
update are float32), so its program keeps the fields it reads in float32, as flow fields are
stored; a float64 run keeps float64.
"""
from __future__ import annotations

import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1602_03643_gb300 import capi
from paper_1602_03643_gb300.driver import IPCSRun
from paper_1602_03643_gb300.guess import GuessNet

NU, DT = 1e-3, 1e-3


def _steps(name, nx, ny, nz=0, **kw):
    c = {"name": name, "what": "steps", "nx": nx, "ny": ny, "nz": nz, "channel": False, "jitter": 0.0,
         "order": "natural", "precision": "mixed", "pc": "amg", "graph": True, "guess": "previous",
         "convection": "abcn", "update": "lumped", "scalars": 0, "batch": True, "host": False, "steps": 2}
    c.update(kw)
    return c


def listed():
    return [
        # a small plane problem in full precision: launches and latency are everything
        _steps("square 32 fp64", 32, 32, precision="fp64", steps=4),
        # a first script: the wrapper's defaults (float64, Jacobi, eager launches), host arrays in
        # and out, the statistics of every step read
        _steps("cube 13 defaults", 13, 12, 11, precision="fp64", pc="jacobi", graph=False, guess="zero",
               host=True, steps=3),
        # a plane problem of working size on a moved mesh, ragged against every tile
        _steps("square 411x389", 411, 389, jitter=0.2, order="rcm", steps=3),
        # the 3D Taylor-Green size: the working set stays in L2; the learned guess runs in the step
        _steps("cube 64 learned", 64, 64, 64, guess="learned", steps=3),
        # wall-bounded flow, periodic in x and z, stretched in y
        _steps("channel 128x95x96", 128, 95, 96, channel=True),
        # the largest runs: a moved mesh in reverse Cuthill-McKee order
        _steps("cube 128 rcm", 128, 128, 128, jitter=0.2, order="rcm"),
        # a mesh generator's order, full precision
        _steps("cube 72 random fp64", 72, 70, 73, jitter=0.2, order="random", precision="fp64"),
        # every option of the scheme: scalars carried along, consistent-mass update
        _steps("cube 48 options", 48, 49, 47, jitter=0.2, order="rcm", scalars=2, update="consistent", steps=3),
        # the Jacobi form of the pressure solve, for users who do without the hierarchy
        _steps("cube 40 jacobi", 40, 40, 40, jitter=0.2, pc="jacobi"),
        # inference and training of the learned guess
        {"name": "guess 96", "what": "guess", "nx": 96, "ny": 96, "nz": 96, "jitter": 0.2, "order": "rcm"},
        {"name": "train 64", "what": "train", "nx": 64, "ny": 64, "nz": 64, "jitter": 0.2, "order": "natural"},
        # products with the constant matrices (post-processing, solvers of the user's own)
        {"name": "products 100", "what": "products", "nx": 100, "ny": 101, "nz": 99, "jitter": 0.2,
         "order": "rcm"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["steps"] * 7 + ["guess", "train", "products"])
    fp64, jacobi = rng.random() < 0.35, rng.random() < 0.25
    plane = what == "steps" and rng.random() < 0.35
    host = rng.random() < 0.2
    # float64 and Jacobi runs take several times as long for the same mesh, host copies as well
    top = 3e4 if fp64 and jacobi else 1e5 if fp64 or jacobi or host else 4e5 if plane else 1.2e6
    dofs = _log_int(rng, 400, top)
    side = dofs ** (0.5 if plane else 1.0 / 3.0)
    n = [max(4, int(round(side * rng.uniform(0.8, 1.25)))) for _ in range(2 if plane else 3)] + [0] * plane
    order, jitter = rng.choice(["natural", "rcm", "rcm", "random"]), rng.choice([0.0, 0.2])
    if what != "steps":
        return {"what": what, "nx": n[0], "ny": n[1], "nz": n[2], "jitter": jitter, "order": order}
    channel = not plane and rng.random() < 0.25
    c = _steps("", *n, channel=channel, jitter=0.0 if channel else jitter, order=order,
               precision="fp64" if fp64 else "mixed", pc="jacobi" if jacobi else "amg",
               graph=rng.random() < 0.75, guess=rng.choice(["zero", "previous", "previous", "learned"]),
               convection="abe" if rng.random() < 0.2 else "abcn",
               update="consistent" if rng.random() < 0.2 else "lumped",
               scalars=rng.choice([0, 0, 0, 1, 2]), batch=rng.random() < 0.9, host=host,
               steps=rng.choice([2, 3]))
    del c["name"]
    return c


# ------------------------------------------------------------------ meshes
def _box(case):
    """Vertices, cells, dof of each vertex, number of dofs, wall dofs and the dof renumbering."""
    n = [case["nx"], case["ny"]] + ([case["nz"]] if case["nz"] else [])
    d = len(n)
    channel = case.get("channel", False)
    axes = [np.linspace(0.0, 1.0, k + 1) for k in n]
    if channel:
        axes[0], axes[2] = 4 * np.pi * axes[0], 4 * np.pi / 3 * axes[2]
        axes[1] = np.tanh(2.0 * (2.0 * axes[1] - 1.0)) / np.tanh(2.0)
    shape = [k + 1 for k in n]
    grid = np.meshgrid(*axes, indexing="ij")
    x = np.stack([g.ravel() for g in grid], axis=1)
    vid = np.arange(x.shape[0], dtype=np.int32).reshape(shape)
    # Kuhn's split of every box: a walk from corner 0 to the opposite one, each order of the axes
    cells = []
    for axis_order in itertools.permutations(range(d)):
        at, walk = [0] * d, []
        for step in (None,) + axis_order:
            if step is not None:
                at[step] = 1
            walk.append(vid[tuple(slice(a, a + k) for a, k in zip(at, n))].ravel())
        cells.append(np.stack(walk, axis=1))
    cells = np.stack(cells, axis=1).reshape(-1, d + 1)
    idx = np.indices(shape).reshape(d, -1)
    wrap = [channel and a != 1 for a in range(d)]
    size = [k if w else k + 1 for k, w in zip(n, wrap)]
    dof = np.zeros(x.shape[0], dtype=np.int64)
    wall = np.zeros(x.shape[0], dtype=bool)
    for a in range(d):
        dof = dof * size[a] + (idx[a] % n[a] if wrap[a] else idx[a])
        if not wrap[a]:
            wall |= (idx[a] == 0) | (idx[a] == n[a])
    n_dofs = int(np.prod(size))
    if case["jitter"]:
        x = _moved(x, cells, ~wall, case["jitter"], n)
    return x, cells, dof.astype(np.int32), n_dofs, np.unique(dof[wall]).astype(np.int32), _order(case, size, wrap)


def _moved(x, cells, inner, frac, n):
    """Inner vertices moved at random; less far where a cell would turn over."""
    g = np.random.default_rng(4)
    shift = torch.from_numpy(g.uniform(-frac, frac, x.shape) / np.array(n) * inner[:, None]).cuda()
    x0, c = torch.from_numpy(x).cuda(), torch.from_numpy(cells).cuda().long()

    def volumes(y):
        return torch.linalg.det(torch.stack([y[c[:, k]] - y[c[:, 0]] for k in range(1, c.shape[1])], dim=1))

    sign = torch.sign(volumes(x0))
    while True:
        bad = volumes(x0 + shift) * sign <= 0
        if not bool(bad.any()):
            return (x0 + shift).cpu().numpy()
        shift[torch.unique(c[bad])] *= 0.5


def _order(case, size, wrap):
    n = int(np.prod(size))
    if case["order"] == "natural":
        return None
    if case["order"] == "random":
        return np.random.default_rng(44).permutation(n).astype(np.int32)
    # reverse Cuthill-McKee on the graph of the split box, level by level
    d = len(size)
    off = [np.array(o) for o in itertools.product((0, 1), repeat=d) if any(o)]
    off = np.array(off + [-o for o in off])
    stride = np.array([int(np.prod(size[a + 1:])) for a in range(d)])

    def neighbours(v):
        p = v[:, None] // stride % np.array(size)
        q = p[:, None, :] + off[None]
        ok = np.ones(q.shape[:2], dtype=bool)
        for a in range(d):
            if wrap[a]:
                q[..., a] %= size[a]
            else:
                ok &= (q[..., a] >= 0) & (q[..., a] < size[a])
        return np.where(ok, q @ stride, -1)

    degree = np.concatenate([(neighbours(b) >= 0).sum(1) for b in np.array_split(np.arange(n), n // 200000 + 1)])
    seen = np.zeros(n, dtype=bool)
    front = np.array([int(np.argmin(degree))])
    seen[front] = True
    levels = [front]
    while front.size:
        q = neighbours(front)
        parent, flat = np.repeat(np.arange(front.size), q.shape[1]), q.ravel()
        keep = (flat >= 0) & ~seen[flat]
        parent, flat = parent[keep], flat[keep]
        flat = flat[np.lexsort((degree[flat], parent))]
        _, first = np.unique(flat, return_index=True)
        front = flat[np.sort(first)]
        seen[front] = True
        levels.append(front)
    perm = np.empty(n, dtype=np.int32)
    perm[np.concatenate(levels)[::-1]] = np.arange(n)
    return perm


class _Mesh:
    """The mesh as the library holds it, with its constant matrices; freed with its last user."""

    def __init__(self, case):
        self.x, self.cells, self.dof, self.n, self.wall, self.perm = _box(case)
        self.dim = self.x.shape[1]
        self.handle = None
        first = np.full(self.n, -1, dtype=np.int64)
        first[self.dof[::-1]] = np.arange(self.dof.size)[::-1]
        self.at = self.x[first]                      # one vertex of every dof

    def open(self):
        if self.handle is None:
            self.handle = capi.oasis_mesh_create(self.dim, self.x, self.cells, self.dof, self.n, self.perm)
            capi.oasis_assemble_constant(self.handle, torch.cuda.current_stream())
        return self

    def __del__(self):
        if self.handle is not None:
            capi.oasis_mesh_destroy(self.handle)


_kept = {}


def _mesh(case):
    key = tuple(case.get(k, False) for k in ("nx", "ny", "nz", "channel", "jitter", "order"))
    if key not in _kept:
        _kept.clear()
        _kept[key] = _Mesh(case)
    return _kept[key]


# ------------------------------------------------------------------ fields
def _fields(case, m, seed):
    """Velocity [d, n] now and one step earlier, pressure [n], scalars [k, n], body force."""
    g = np.random.default_rng(seed)
    lo, hi = m.at.min(0), m.at.max(0)
    xi = (m.at - lo) / (hi - lo)
    d = m.dim

    def wave():
        k = g.integers(1, 3, d) * g.choice([-1, 1], d)
        return k, np.cos(2 * np.pi * (xi @ k) + g.uniform(0, 2 * np.pi))

    if case["channel"]:
        u = np.zeros((d, m.n))
        u[0] = 90.0 * (1.0 - m.at[:, 1] ** 2)
        inner = np.ones(m.n, dtype=bool)
        inner[m.wall] = False
        u[:, inner] += 9.0 * g.uniform(-1.0, 1.0, (d, int(inner.sum())))
        u[:, m.wall] = 0.0
        before, p, force = u.copy(), np.zeros(m.n), (1.0, 0.0, 0.0)
    else:
        u = np.zeros((d, m.n))                       # a few solenoidal waves
        for _ in range(4):
            k, c = wave()
            q = k / (hi - lo)
            a = g.normal(size=d)
            a -= q * (a @ q) / (q @ q)
            u += 0.6 * a[:, None] / np.linalg.norm(a) * c
        before, p, force = 1.001 * u, 0.25 * wave()[1] + 0.1 * wave()[1], (0.0,) * d
    c = np.stack([wave()[1] + 0.05 * g.uniform(-1, 1, m.n) for _ in range(case["scalars"])]) if case["scalars"] else None
    return u, before, p, c, force


_DIFF, _SRC = (1e-3, 2e-2), (0.0, 0.5)


def _params(n, seed):
    """Network parameters of the size that training leaves."""
    g = np.random.default_rng(seed)
    h = 32
    return np.concatenate([g.normal(size=6 * h) * 0.58, 0.1 * g.normal(size=h), g.normal(size=2 * h * h) * 0.18,
                           0.1 * g.normal(size=h), 0.02 * g.normal(size=h), [0.01], [1.0, -0.1]]).astype(np.float32)


class _State:
    solver = net = run = None

    def __del__(self):
        if self.solver is not None:
            capi.oasis_solver_destroy(self.solver)
        self.solver = self.mesh = None


def prepare(case, seed):
    m = _mesh(case).open()
    s = _State()
    s.case, s.mesh = case, m
    if case["what"] != "steps":
        gen = torch.Generator("cuda").manual_seed(int(seed))
        if case["what"] == "products":
            s.x = torch.randn(m.n, dtype=torch.float64, device="cuda", generator=gen)
            s.x32 = s.x.float()
            s.y = [torch.empty_like(s.x), torch.empty_like(s.x32), torch.empty_like(s.x),
                   torch.empty(1, dtype=torch.float64, device="cuda")]
            return s
        s.x = torch.randn(m.n, 3, device="cuda", generator=gen)
        s.t = s.x[:, 1] + 0.1 * torch.randn(m.n, device="cuda", generator=gen)
        s.y = torch.empty(m.n, device="cuda")
        s.net = GuessNet(m.handle, m.n, params=_params(m.n, seed))
        return s
    fp64 = case["precision"] == "fp64"
    rtol = 1e-12 if fp64 else 1e-8
    opt = dict(precision=capi.OASIS_FP64 if fp64 else capi.OASIS_MIXED, rtol_u=rtol, rtol_p=rtol, max_it_u=5000,
               max_it_p=50000, batch_rhs=int(case["batch"]), use_graph=int(case["graph"]),
               guess={"zero": capi.OASIS_GUESS_ZERO, "previous": capi.OASIS_GUESS_PREV_PHI,
                      "learned": capi.OASIS_GUESS_LEARNED}[case["guess"]],
               pressure_pc=capi.OASIS_PC_AMG if case["pc"] == "amg" else capi.OASIS_PC_JACOBI,
               convection=capi.OASIS_CONV_ABE if case["convection"] == "abe" else capi.OASIS_CONV_ABCN,
               velocity_update=capi.OASIS_UPDATE_CONSISTENT if case["update"] == "consistent"
               else capi.OASIS_UPDATE_LUMPED)
    u, before, p, c, force = _fields(case, m, seed)
    g = np.ascontiguousarray(u[:, m.wall])
    ns = case["scalars"]
    gc = np.ascontiguousarray(c[:, m.wall]) if ns else None
    if case["host"]:
        scal = SimpleNamespace(c0=c, diffusivity=np.array(_DIFF[:ns]), source=np.array(_SRC[:ns]), dirichlet=m.wall,
                               g=lambda t: gc) if ns else None
        mesh = SimpleNamespace(dim=m.dim, coords=m.x, cells=m.cells, dof_of_vertex=m.dof, n_dofs=m.n)
        s.run = IPCSRun(SimpleNamespace(mesh=mesh, nu=NU, dt=DT, f=force, dirichlet=m.wall, u_nm1=u, u_nm2=before, p=p,
                                        t0=0.0, g=lambda t: g, perm=m.perm, scalars=scal), **opt)
        if case["guess"] == "learned":
            s.net = GuessNet(s.run.mesh, m.n, params=_params(m.n, 1))
            s.run.attach_guess_net(s.net)
        return s
    stream = torch.cuda.current_stream()
    s.solver = capi.oasis_solver_create(m.handle, capi.make_params(NU, DT, force, **opt), m.wall, stream)
    if case["guess"] == "learned":
        s.net = GuessNet(m.handle, m.n, params=_params(m.n, 1))
        capi.oasis_solver_set_guess_net(s.solver, s.net.handle)
    if ns:
        capi.oasis_solver_set_scalars(s.solver, _DIFF[:ns], _SRC[:ns], m.wall)
        s.c, s.gc = torch.from_numpy(c).cuda(), torch.from_numpy(gc).cuda()
    s.u1, s.u2, s.p, s.g = (torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (u, before, p, g))
    s.u_out, s.p_out = torch.empty_like(s.u1), torch.empty_like(s.p)
    s.c_out = torch.empty_like(s.c) if ns else None
    return s


def run(s):
    case, m = s.case, s.mesh
    stream = torch.cuda.current_stream()
    if case["what"] == "products":
        y = s.y
        capi.oasis_spmv_f64(m.handle, capi.OASIS_MAT_M, s.x, y[0], 0, stream)
        capi.oasis_spmv_f32(m.handle, capi.OASIS_MAT_K, s.x32, y[1], 0, stream)
        capi.oasis_spmv_dot_f64(m.handle, capi.OASIS_MAT_K, s.x, y[2], y[3], stream)
        return list(y)
    if case["what"] == "guess":
        return s.net.forward(s.x, s.y)
    if case["what"] == "train":
        return list(s.net.loss_and_grad(s.x, s.t))
    if case["host"]:
        r, pb = s.run, s.run.pb
        capi.oasis_set_fields(r.solver, pb.u_nm1, pb.u_nm2, pb.p, 0.0, False, r.stream)
        if case["scalars"]:
            capi.oasis_set_scalar_fields(r.solver, pb.scalars.c0, False, r.stream)
        r.t, r.stats = 0.0, []
        r.step(case["steps"])
        u, p, _ = r.fields()
        out = [u, p] + ([r.scalar_fields()] if case["scalars"] else [])
        return out if case["precision"] == "fp64" else [v.astype(np.float32) for v in out]
    capi.oasis_set_fields(s.solver, s.u1, s.u2, s.p, 0.0, True, stream)
    if case["scalars"]:
        capi.oasis_set_scalar_fields(s.solver, s.c, True, stream)
        capi.oasis_set_scalar_dirichlet(s.solver, s.gc, True, stream)
    for _ in range(case["steps"]):
        capi.oasis_set_dirichlet(s.solver, s.g, True, stream)
        capi.oasis_step(s.solver, stream, want_stats=False)
    capi.oasis_get_fields(s.solver, m.dim, m.n, True, s.u_out, s.p_out, None, stream)
    out = [s.u_out, s.p_out]
    if case["scalars"]:
        capi.oasis_get_scalar_fields(s.solver, case["scalars"], m.n, True, s.c_out, stream)
        out.append(s.c_out)
    return out if case["precision"] == "fp64" else [v.float() for v in out]


# ------------------------------------------------------------------ work
def work(case):
    """Bytes and operations of one pass: inputs, outputs, the mesh and its matrices once per step;
    per step one product with every matrix that the step has (its solves repeat theirs as often
    as the data ask for)."""
    d = 3 if case["nz"] else 2
    n = np.prod([k + 1.0 for k in (case["nx"], case["ny"], case["nz"]) if k])
    cells = (6.0 if d == 3 else 2.0) * np.prod([float(k) for k in (case["nx"], case["ny"], case["nz"]) if k])
    nnz = (15.0 if d == 3 else 7.0) * n
    if case["what"] == "products":
        return {"bytes": float(nnz * (8 + 4 + 8 + 12) + n * (16 + 8 + 16)), "flops": float(6 * nnz)}
    if case["what"] == "guess":
        return {"bytes": float(4 * nnz + n * (12 + 4)), "flops": float(n * (2 * 192 + 2 * 2048 + 70) + 35 * nnz * 2)}
    if case["what"] == "train":
        return {"bytes": float(4 * nnz + n * (12 + 4) + 2340 * 4),
                "flops": float(3 * n * (2 * 192 + 2 * 2048 + 70) + 70 * nnz * 2)}
    v = 8.0 if case["precision"] == "fp64" else 4.0
    k = case["scalars"]
    mats = nnz * (v * (2 + d) + 4) + cells * (4 * (d + 1) + v * d * (d + 1))
    step = mats + n * 8 * (2 * d + 1 + d + 1 + 2 * k)
    flops = 2 * nnz * (2 * d + 1 + d + d + 2 * k) + cells * 2 * d * (d + 1)
    return {"bytes": float(case["steps"] * step), "flops": float(case["steps"] * flops)}


# ------------------------------------------------------------------ 64-bit values
class _Operators:
    """Mass, stiffness, derivative and convection matrices of linear elements on the mesh, float64."""

    def __init__(self, m):
        dev = "cuda"
        self.n, self.d = m.n, m.dim
        d = m.dim
        x = torch.from_numpy(m.x).to(dev)
        cv = torch.from_numpy(m.cells).to(dev).long()
        self.c = torch.from_numpy(m.dof).to(dev).long()[cv]
        J = torch.stack([x[cv[:, k]] - x[cv[:, 0]] for k in range(1, d + 1)], dim=2)
        self.vol = torch.linalg.det(J).abs() / math.factorial(d)
        g = torch.linalg.inv(J)
        self.g = torch.cat([-g.sum(1, keepdim=True), g], dim=1)          # [cells, d + 1, d]
        self.pairs = [(a, b) for a in range(d + 1) for b in range(d + 1)]
        key = torch.cat([self.c[:, a] * self.n + self.c[:, b] for a, b in self.pairs])
        uniq, self.to = torch.unique(key, return_inverse=True)
        self.row, self.col = uniq // self.n, uniq % self.n
        self.ptr = torch.zeros(self.n + 1, dtype=torch.long, device=dev)
        self.ptr[1:] = torch.cumsum(torch.bincount(self.row, minlength=self.n), 0)
        self.nnz = uniq.numel()
        self.M = self.summed(lambda a, b: self.vol * ((2.0 if a == b else 1.0) / ((d + 1) * (d + 2))))
        self.K = self.summed(lambda a, b: self.vol * (self.g[:, a] * self.g[:, b]).sum(1))
        self.G = [self.summed(lambda a, b, k=k: self.vol * self.g[:, b, k] / (d + 1)) for k in range(d)]
        self.ML = self.mul(self.M, torch.ones(self.n, dtype=torch.float64, device=dev))

    def summed(self, part):
        out = torch.zeros(self.nnz, dtype=torch.float64, device=self.vol.device)
        t = self.vol.numel()
        for q, (a, b) in enumerate(self.pairs):
            out.index_add_(0, self.to[q * t:(q + 1) * t], part(a, b))
        return out

    def convection(self, u):                                             # u [n, d]
        d = self.d
        ue = u[self.c]
        total = ue.sum(1)
        w = self.vol / ((d + 1) * (d + 2))
        return self.summed(lambda a, b: w * (self.g[:, b] * (total + ue[:, a])).sum(1))

    def mul(self, v, x):
        m = torch.sparse_csr_tensor(self.ptr, self.col, v, (self.n, self.n))
        return m @ x

    def diag(self, v):
        out = torch.zeros(self.n, dtype=torch.float64, device=v.device)
        on = self.row == self.col
        out[self.row[on]] = v[on]
        return out

    def with_unit_rows(self, v, fixed):
        v = v.clone()
        v[fixed[self.row]] = 0.0
        v[fixed[self.row] & (self.row == self.col)] = 1.0
        return v


def _solve(mul, b, dinv, symmetric, tol=2e-14, most=6000):
    """Jacobi-preconditioned CG or BiCGStab on the columns of b together, started again from the true residual."""
    x = torch.zeros_like(b)
    bb = b.norm(dim=0)
    bb = torch.where(bb > 0, bb, torch.ones_like(bb))
    best, best_x = math.inf, x
    tiny = 1e-300
    for _ in range(8):
        r = b - mul(x)
        far = float((r.norm(dim=0) / bb).max())
        if far < best:
            best, best_x = far, x.clone()
        elif far > 0.5 * best:
            break
        if far <= tol:
            break
        aim, start = r.norm(dim=0) * 1e-7, r.clone()
        y = torch.zeros_like(b)
        if symmetric:
            z = dinv * r
            p, rz = z.clone(), (r * z).sum(0)
            for it in range(most):
                q = mul(p)
                al = rz / ((p * q).sum(0) + tiny)
                y += al * p
                r -= al * q
                z = dinv * r
                new = (r * z).sum(0)
                p = z + new / (rz + tiny) * p
                rz = new
                if it % 16 == 15 and bool((r.norm(dim=0) <= aim).all()):
                    break
        else:
            p, v = torch.zeros_like(r), torch.zeros_like(r)
            rho = al = om = torch.ones_like(bb)
            live = torch.ones_like(bb, dtype=torch.bool)
            for it in range(most):
                new = (start * r).sum(0)
                p = r + new / (rho + tiny) * (al / (om + tiny)) * (p - om * v)
                rho = torch.where(live, new, rho)
                ph = dinv * p
                v = mul(ph)
                al = torch.where(live, rho / ((start * v).sum(0) + tiny), torch.zeros_like(al))
                s = r - al * v
                sh = dinv * s
                t = mul(sh)
                om = torch.where(live, (t * s).sum(0) / ((t * t).sum(0) + tiny), torch.zeros_like(om))
                y += al * ph + om * sh
                r = torch.where(live, s - om * t, r)
                live = live & (r.norm(dim=0) > aim)
                if not bool(live.any()):
                    break
        x = x + y
    return best_x


def _exact_steps(case, m, seed):
    o = _Operators(m)
    d, n, dev = m.dim, m.n, "cuda"
    u, before, p, c, force = _fields(case, m, seed)
    u1, u2 = torch.from_numpy(u).to(dev).T.contiguous(), torch.from_numpy(before).to(dev).T.contiguous()
    p = torch.from_numpy(p).to(dev)
    fixed = torch.zeros(n, dtype=torch.bool, device=dev)
    fixed[torch.from_numpy(m.wall).to(dev).long()] = True
    held = u1.clone()
    f = torch.tensor(force, dtype=torch.float64, device=dev)
    ns = case["scalars"]
    cs = torch.from_numpy(c).to(dev).T.contiguous() if ns else None
    c_held = cs.clone() if ns else None
    dk = o.diag(o.K)[:, None]
    for _ in range(case["steps"]):
        C = o.convection(1.5 * u1 - 0.5 * u2)
        grad_p = torch.stack([o.mul(o.G[k], p) for k in range(d)], 1)
        if case["convection"] == "abe":
            A = o.M / DT + 0.5 * NU * o.K
            r0 = -NU * o.mul(o.K, u1) - 1.5 * o.mul(o.convection(u1), u1) + 0.5 * o.mul(o.convection(u2), u2)
        else:
            A = o.M / DT + 0.5 * C + 0.5 * NU * o.K
            r0 = -o.mul(C + NU * o.K, u1)
        r0 = r0 + o.ML[:, None] * f - grad_p
        r0[fixed] = (held - u1)[fixed]
        A = o.with_unit_rows(A, fixed)
        ui = u1 + _solve(lambda v: o.mul(A, v), r0, 1.0 / o.diag(A)[:, None], False)
        b = -sum(o.mul(o.G[k], ui[:, k].contiguous()) for k in range(d))[:, None] / DT
        b = b - b.mean()
        phi = _solve(lambda v: o.mul(o.K, v), b, 1.0 / dk, True)[:, 0]
        push = -DT * torch.stack([o.mul(o.G[k], phi) for k in range(d)], 1)
        if case["update"] == "consistent":
            known = torch.where(fixed[:, None], held - ui, torch.zeros_like(ui))
            rhs = torch.where(fixed[:, None], torch.zeros_like(ui), push - o.mul(o.M, known))
            keep = (~fixed)[:, None]
            step = _solve(lambda v: torch.where(keep, o.mul(o.M, v), v), rhs, 1.0 / o.diag(o.M)[:, None], True) + known
        else:
            step = push / o.ML[:, None]
        un = ui + step
        un[fixed] = held[fixed]
        for a in range(ns):
            B = o.with_unit_rows(o.M / DT + 0.5 * C + 0.5 * _DIFF[a] * o.K, fixed)
            r = -o.mul(C + _DIFF[a] * o.K, cs[:, a].contiguous()) + _SRC[a] * o.ML
            r[fixed] = (c_held - cs)[fixed, a]
            cs[:, a] += _solve(lambda v: o.mul(B, v), r[:, None], 1.0 / o.diag(B)[:, None], False)[:, 0]
            cs[fixed, a] = c_held[fixed, a]
        p = p + phi
        p = p - p.mean()
        u1, u2 = un, u1
    return [u1.T.contiguous(), p] + ([cs.T.contiguous()] if ns else [])


def _exact_net(o, x, t, params, train):
    """The network in float64 with its weights on the bfloat16 grid; loss and gradient when training."""
    w = torch.from_numpy(params).cuda().bfloat16().double().requires_grad_(train)
    h = 32
    w1a, w1b, c1 = w[:96].view(h, 3), w[96:192].view(h, 3), w[192:224]
    w2a, w2b, c2 = w[224:1248].view(h, h), w[1248:2272].view(h, h), w[2272:2304]
    w3, c3, skip = w[2304:2336], w[2336], w[2337:2339]
    off = o.row != o.col
    row, col = o.row[off], o.col[off]
    degree = torch.bincount(row, minlength=o.n).clamp(min=1).double()[:, None]

    def mean(v):
        return torch.zeros(o.n, v.shape[1], dtype=v.dtype, device=v.device).index_add(0, row, v[col]) / degree

    h1 = torch.relu(x @ w1a.T + mean(x) @ w1b.T + c1)
    h2 = torch.relu(h1 @ w2a.T + mean(h1) @ w2b.T + c2)
    y = h2 @ w3 + c3 + x[:, 1:] @ skip
    if not train:
        return y
    loss = ((y - t) ** 2).mean()
    loss.backward()
    return [loss.detach().view(1), w.grad]


def exact(case, seed):
    m = _mesh(case)
    if case["what"] == "steps":
        out = _exact_steps(case, m, seed)
        return [v.cpu().numpy() for v in out] if case["host"] else out
    o = _Operators(m)
    gen = torch.Generator("cuda").manual_seed(int(seed))
    # these entry points take vectors in the library's own order of the dofs
    at = torch.arange(m.n, device="cuda") if m.perm is None else torch.from_numpy(m.perm).cuda().long()

    def back(v):
        out = torch.empty_like(v)
        out[at] = v
        return out

    if case["what"] == "products":
        x = torch.randn(m.n, dtype=torch.float64, device="cuda", generator=gen)
        x32, x = x.float().double()[at], x[at]
        kx = o.mul(o.K, x)
        return [back(o.mul(o.M, x)), back(o.mul(o.K, x32)), back(kx), (x @ kx).view(1)]
    x = torch.randn(m.n, 3, device="cuda", generator=gen)
    t = x[:, 1] + 0.1 * torch.randn(m.n, device="cuda", generator=gen)
    y = _exact_net(o, x.double()[at], t.double()[at], _params(m.n, seed), case["what"] == "train")
    return y if case["what"] == "train" else back(y)
