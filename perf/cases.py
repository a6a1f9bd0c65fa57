"""The work that is timed: calls a user of the library makes, over the sizes, degrees and precisions that it serves.

Kinds of case (``"kind"``), each through the public Python entry points:

* ``apply``     one operator application of a caller's own Krylov method;
* ``vcycle``    one multigrid V-cycle (the library as a preconditioner);
* ``solve``     a whole Poisson solve: CG with a V-cycle, or full multigrid with patch smoothing;
* ``gradient``  one step of a coefficient identification: J(kappa) and dJ/dkappa through autograd, a new kappa each time;
* ``batch``     many small independent problems in one launch.

The mesh is UnitCubeMesh(n0 * 2^refine) with Lagrange degree 1, 2 or 3; kappa is 1 or a log-normal random field.
``exact`` restates the discretisation in torch FP64 on the lattice of the degrees of freedom.
"""
import itertools
import math

import numpy as np
import torch

import paper_2104_08012_gb300 as fe
from paper_2104_08012_gb300.autograd import poisson_objective

DEV = "cuda"
DTYPES = {"f64": (fe.FE_F64, torch.float64), "f32": (fe.FE_F32, torch.float32), "bf16": (fe.FE_BF16, torch.float32)}
PRECISIONS = {"f64": fe.FE_PREC_F64, "mixed_f32": fe.FE_PREC_MIXED_F32, "mixed_bf16": fe.FE_PREC_MIXED_BF16}


def listed():
    return [
        # the smallest call: one application on a mesh of a unit test or of a coarse level; launch latency
        _apply(1, 8, "f64", "field", "apply_p1_f64_n8"),
        # the operator of the headline problem (kappa = 1)
        _apply(2, 64, "f64", "one", "apply_p2_f64_n64"),
        # an odd size with a varying coefficient
        _apply(2, 45, "f64", "field", "apply_p2_f64_n45_field"),
        # single precision, far larger than the caches
        _apply(2, 128, "f32", "one", "apply_p2_f32_n128"),
        # the paper's degree
        _apply(3, 32, "f64", "field", "apply_p3_f64_n32_field"),
        # the V-cycle as preconditioner of a caller's Krylov method, a size that is no power of two
        {"name": "vcycle_p2_f64_n40_field", "kind": "vcycle", "degree": 2, "n0": 5, "refine": 3, "dtype": "f64",
         "kappa": "field"},
        # a small solve: many launches on little data; load vector by quadrature
        _solve(1, 4, 2, "f64", "field", "quad", "solve_p1_f64_n16_field"),
        # the headline benchmark
        _solve(2, 8, 3, "f64", "one", "nodal", "solve_p2_f64_n64"),
        # mixed precision at the size where it is meant to be used
        _solve(2, 8, 4, "mixed_f32", "one", "nodal", "solve_p2_mixed_f32_n128"),
        # the paper's own solver: P3, full multigrid, vertex-star patches
        dict(_solve(3, 4, 3, "f64", "one", "nodal", "solve_p3_fmg_patch_n32"), method="fmg_patch"),
        # one step of a coefficient identification on P1 96^3
        {"name": "gradient_p1_n96", "kind": "gradient", "degree": 1, "n0": 12, "refine": 3},
        # many independent problems, P1 and P2 mixed, 16^3 to 48^3
        {"name": "batch_64", "kind": "batch", "problems": 64},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def hierarchy(degree, lo, hi):  # a small direct coarse solve, refined to a size in [lo, hi]
        while True:
            n0, refine = rng.randint(2, {1: 12, 2: 8, 3: 5}[degree]), rng.randint(1, 4)
            if lo <= n0 << refine <= hi:
                return n0, refine

    kappa = rng.choice(["one", "field"])
    kind = rng.choice(["apply", "apply", "vcycle", "solve", "solve", "gradient", "batch"])
    if kind == "apply":
        degree = rng.choice([1, 2, 2, 3])
        dtype = rng.choice(["f64", "f64", "f32", "bf16"])
        n = size(8, {1: 128, 2: 96, 3: 40}[degree])
        return _apply(degree, n, dtype, kappa)
    if kind == "vcycle":
        degree = rng.choice([1, 2, 2, 3])
        n0, refine = hierarchy(degree, 8, {1: 112, 2: 80, 3: 32}[degree])
        return {"kind": kind, "degree": degree, "n0": n0, "refine": refine, "dtype": rng.choice(["f64", "f64", "f32"]),
                "kappa": kappa}
    if kind == "solve":
        degree = rng.choice([1, 2, 2, 3])
        n0, refine = hierarchy(degree, 8, {1: 96, 2: 64, 3: 32}[degree])
        precision = rng.choice(["f64", "f64", "mixed_f32", "mixed_bf16"])
        rhs = "quad" if (n0 << refine) <= 24 else "nodal"
        case = _solve(degree, n0, refine, precision, kappa, rhs)
        if degree > 1 and precision == "f64" and rng.random() < 0.25:
            case["method"] = "fmg_patch"
        return case
    if kind == "gradient":
        n0, refine = hierarchy(1, 16, 96)
        return {"kind": kind, "degree": 1, "n0": n0, "refine": refine}
    return {"kind": "batch", "problems": size(4, 60)}


def _apply(degree, n, dtype, kappa, name=None):
    return {**({"name": name} if name else {}), "kind": "apply", "degree": degree, "n0": n, "refine": 0,
            "dtype": dtype, "kappa": kappa}


def _solve(degree, n0, refine, precision, kappa, rhs, name=None):
    return {**({"name": name} if name else {}), "kind": "solve", "degree": degree, "n0": n0, "refine": refine,
            "precision": precision, "kappa": kappa, "rhs": rhs, "method": "cg"}


# ------------------------------------------------------------------ inputs
PERMS = list(itertools.permutations(range(3)))  # the six Kuhn tets of a cube, cells 6q .. 6q+5


def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(1_000_003 * (seed + 1) + salt)


def _centroids(n):
    """Cell centroids, [6 n^3, 3], cubes x fastest."""
    r = torch.arange(n, device=DEV, dtype=torch.float64)
    z, y, x = torch.meshgrid(r, r, r, indexing="ij")
    base = torch.stack([x, y, z], -1).reshape(-1, 1, 3)
    off = torch.zeros(6, 3, dtype=torch.float64)
    for t, p in enumerate(PERMS):
        for k, a in enumerate(p):
            off[t, a] = (3 - k) / 4
    return ((base + off.to(DEV)) / n).reshape(-1, 3)


def _field(points, seed, salt, features=64, length=0.2):
    """Log-normal random field exp(g) by random Fourier features (sigma = 1, correlation length 0.2)."""
    g = _gen(seed, salt)
    omega = torch.randn(features, 3, generator=g, device=DEV, dtype=torch.float64) / length
    phase = torch.rand(features, generator=g, device=DEV, dtype=torch.float64) * 2 * math.pi
    out = torch.empty(points.shape[0], dtype=torch.float64, device=DEV)
    for s in range(0, points.shape[0], 1 << 20):
        out[s:s + (1 << 20)] = torch.cos(points[s:s + (1 << 20)] @ omega.T + phase).sum(1)
    return torch.exp(out * math.sqrt(2.0 / features))


def _kappa(case, n, seed, salt=7):
    return _field(_centroids(n), seed, salt) if case["kappa"] == "field" else None


def _waves(points, seed, salt):
    """A smooth right-hand side or target: the sin product and eight seeded low-frequency sine products."""
    g = _gen(seed, salt)
    amp = torch.randn(8, generator=g, device=DEV, dtype=torch.float64)
    freq = torch.randint(1, 4, (8, 3), generator=g, device=DEV).to(torch.float64)
    out = 3 * math.pi ** 2 * torch.sin(math.pi * points).prod(-1)
    for a, p in zip(amp, freq):
        out += a * torch.sin(math.pi * p * points).prod(-1)
    return out


def _random(n, seed, salt, dtype=torch.float64):
    return (torch.rand(n, generator=_gen(seed, salt), device=DEV, dtype=torch.float64) * 2 - 1).to(dtype)


def _gauss_points():
    """The 27-point conical rule of FE_RHS_QUAD_F on the reference tet: points [27, 3] and weights."""
    x, w = np.polynomial.legendre.leggauss(3)
    x, w = (x + 1) / 2, w / 2
    pts, wts = [], []
    for (u, a), (v, b), (s, c) in itertools.product(zip(x, w), zip(x, w), zip(x, w)):
        pts.append((u, (1 - u) * v, (1 - u) * (1 - v) * s))
        wts.append(a * b * c * (1 - u) ** 2 * (1 - v))
    return np.array(pts), np.array(wts)


def _quadrature_points(n):
    """Physical quadrature points of every cell, [6 n^3, 27, 3]."""
    xi, _ = _gauss_points()
    r = torch.arange(n, device=DEV, dtype=torch.float64)
    z, y, x = torch.meshgrid(r, r, r, indexing="ij")
    base = torch.stack([x, y, z], -1).reshape(-1, 1, 1, 3)
    off = np.zeros((6, 27, 3))
    for t, p in enumerate(PERMS):
        # vertex j of the tet is the sum of the first j unit steps, so step k enters with xi_k + xi_k+1 + ...
        for k, a in enumerate(p):
            off[t, :, a] = xi[:, k:].sum(1)
    return ((base + torch.from_numpy(off).to(DEV)[None]) / n).reshape(-1, 27, 3)


def _order(n, k):
    """Lattice index (x fastest, (kn+1)^3 points) of every dof, in the library's dof order."""
    m = k * n + 1
    lat = torch.arange(m ** 3, device=DEV).reshape(m, m, m)
    if k != 2:
        return lat.reshape(-1)
    par = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 0), (1, 0, 1), (0, 1, 1), (1, 1, 1)]
    return torch.cat([lat[pz::2, py::2, px::2].reshape(-1) for px, py, pz in par])


def _coords(n, k):
    """Coordinates of the dofs, [(kn+1)^3, 3]."""
    m = k * n + 1
    i = _order(n, k)
    return torch.stack([i % m, (i // m) % m, i // (m * m)], -1).to(torch.float64) / (k * n)


def _batch_table(count, seed):
    r = np.random.default_rng(seed + 2)
    sizes = r.choice([16, 24, 32, 40, 48], size=count)
    degrees = np.array([1] * (count // 2) + [2] * (count - count // 2))
    r.shuffle(degrees)
    return [(int(n), int(d)) for n, d in zip(sizes, degrees)]


BATCH_SIZES_SEED = 21040801  # the mesh sizes and degrees of a batch are the case's; kappa and f are the seed's


def _load_input(case, n, seed):
    pts = _quadrature_points(n) if case["rhs"] == "quad" else _coords(n, case["degree"])
    return _waves(pts, seed, 11).contiguous()


# -------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        table = _batch_table(case["problems"], BATCH_SIZES_SEED)
        batch = fe.Batch([(n // 8, 3, k) for n, k in table])
        f, u = [], []
        for p, ((n, k), h) in enumerate(zip(table, batch.problems)):
            h.set_coefficient(_field(_centroids(n), seed, 100 + p))
            f.append(_waves(_coords(n, k), seed, 300 + p))
            u.append(torch.empty(h.n_dofs(), dtype=torch.float64, device=DEV))
        return {"kind": kind, "batch": batch, "f": f, "u": u}
    n = case["n0"] << case["refine"]
    h = fe.Hierarchy(case["n0"], case["refine"], case["degree"])
    s = {"kind": kind, "h": h}
    dofs = h.n_dofs()
    if kind == "gradient":
        pts = _coords(n, 1)
        return {**s, "kappa": _field(_centroids(n), seed, 7), "f": torch.ones(dofs, dtype=torch.float64, device=DEV),
                "target": _waves(pts, seed, 13) / 100, "opts": fe.default_opts(rtol=1e-10)}
    kappa = _kappa(case, n, seed)
    if kappa is not None:
        h.set_coefficient(kappa)
    if kind in ("apply", "vcycle"):
        dtype, store = DTYPES[case["dtype"]]
        x = _random(dofs, seed, 3, store)
        if kind == "vcycle":  # a residual: zero on the boundary rows
            x[torch.from_numpy(h.boundary_mask()).to(DEV)] = 0
        return {**s, "dtype": dtype, "x": x, "y": torch.empty_like(x)}
    s["f"] = _load_input(case, n, seed)
    s["rhs"] = fe.FE_RHS_QUAD_F if case["rhs"] == "quad" else fe.FE_RHS_NODAL_F
    s["u"] = torch.empty(dofs, dtype=torch.float64, device=DEV)
    if case["method"] == "fmg_patch":
        h.set_smoother(fe.FE_SMOOTHER_PATCH)
        s["opts"] = fe.default_opts(precond=fe.FE_PC_FMG, max_it=2)
    else:
        s["opts"] = fe.default_opts(rtol=1e-8, precision=PRECISIONS[case["precision"]])
    return s


def run(state):
    kind = state["kind"]
    if kind == "apply":
        return state["h"].apply_operator(state["x"], state["y"], dtype=state["dtype"])
    if kind == "vcycle":
        return state["h"].vcycle(state["x"], state["y"], dtype=state["dtype"])
    if kind == "solve":
        state["h"].solve(state["f"], state["u"], rhs_kind=state["rhs"], opts=state["opts"])
        return state["u"]
    if kind == "gradient":
        kappa = state["kappa"].detach().clone().requires_grad_()
        J = poisson_objective(kappa, state["h"], state["f"], state["target"], opts=state["opts"])
        J.backward()
        return {"J": J.detach(), "gradient": kappa.grad}
    state["batch"].solve(state["f"], state["u"], rtol=1e-8)
    return state["u"]


# ------------------------------------------------------------------- work
ROW = {1: 7, 2: 25, 3: 47}  # entries of an assembled row, on average


def _work(kind, degree, n, iterations, value, field):
    dofs, cells = (degree * n + 1) ** 3, 6 * n ** 3
    cycle = 2 * 6 * ROW[degree] * dofs * 8 / 7  # six operator-like passes on every level
    io = 2 * value * dofs + (value * cells if field else 0)
    if kind == "apply":
        return {"bytes": io, "flops": 2 * ROW[degree] * dofs}
    return {"bytes": io, "flops": iterations * cycle}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        parts = [_work(kind, k, n, 10, 8, True) for n, k in _batch_table(case["problems"], BATCH_SIZES_SEED)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    n, degree = case["n0"] << case["refine"], case["degree"]
    if kind == "gradient":
        w = _work(kind, degree, n, 2 * 11, 8, True)
        return {"bytes": w["bytes"] + 8 * 6 * n ** 3, "flops": w["flops"]}
    value = 8 if case.get("dtype", "f64") == "f64" else 4
    w = _work(kind, degree, n, 1 if kind == "vcycle" else 10, value, case["kappa"] == "field")
    if kind == "solve" and case["rhs"] == "quad":
        w["bytes"] += 8 * 27 * 6 * n ** 3 - 8 * (degree * n + 1) ** 3
    return w


# ------------------------------------------------- the same in torch, FP64
def _basis(k):
    """Monomial exponents and coefficients [basis, monomial] of the P_k Lagrange basis; nodes times k as (L0..L3)."""
    expo = [(a, b, c) for a in range(k + 1) for b in range(k + 1 - a) for c in range(k + 1 - a - b)]
    nodes = np.array(expo, dtype=np.float64) / k
    vander = np.array([[np.prod([p[i] ** e[i] for i in range(3)]) for e in expo] for p in nodes])
    return expo, np.linalg.inv(vander).T


def _moment(a, b, c):
    f = math.factorial
    return f(a) * f(b) * f(c) / f(a + b + c + 3)


def _reference(k):
    """Reference mass [nd, nd] and derivative products [3, 3, nd, nd] of the P_k basis."""
    expo, coef = _basis(k)
    nd = len(expo)

    def product(da, db):
        out = np.zeros((nd, nd))
        for i, e in enumerate(expo):
            for j, f in enumerate(expo):
                e2, f2, w = list(e), list(f), 1.0
                if da is not None:
                    w, e2[da] = w * e[da], e2[da] - 1
                if db is not None:
                    w, f2[db] = w * f[db], f2[db] - 1
                if w:
                    out[i, j] = w * _moment(*(p + q for p, q in zip(e2, f2)))
        return coef @ out @ coef.T

    return product(None, None), np.array([[product(a, b) for b in range(3)] for a in range(3)])


class _Lattice:
    """-div(kappa grad) with Dirichlet elimination, cell by cell on strided slices of the dof lattice."""

    def __init__(self, n, k, kappa):
        self.n, self.k, self.m = n, k, k * n + 1
        expo, coef = _basis(k)
        mass, stiff = _reference(k)
        self.offsets, self.K = [], []
        for p in PERMS:
            J = np.zeros((3, 3))
            for col in range(3):
                for a in p[:col + 1]:
                    J[a, col] = 1.0
            G = np.linalg.inv(J) @ np.linalg.inv(J).T / n
            self.K.append(torch.from_numpy(np.einsum("ab,abij->ij", G, stiff)).to(DEV))
            self.offsets.append([tuple(int(v) for v in np.rint(J @ np.array(e, dtype=float))) for e in expo])
        self.M = torch.from_numpy(mass / n ** 3).to(DEV)
        self.coef, self.expo = coef, expo
        self.kappa = None if kappa is None else kappa.reshape(-1, 6).T.contiguous()
        inner = torch.zeros(self.m, self.m, self.m, dtype=torch.bool, device=DEV)
        inner[1:-1, 1:-1, 1:-1] = True
        self.inner, self.order = inner, _order(n, k)

    def _view(self, u, o):
        e = self.k * (self.n - 1) + 1
        return u[o[2]:o[2] + e:self.k, o[1]:o[1] + e:self.k, o[0]:o[0] + e:self.k]

    def _gather(self, u, t):
        return torch.stack([self._view(u, o).reshape(-1) for o in self.offsets[t]])

    def _scatter(self, y, t, part):
        for row, o in zip(part, self.offsets[t]):
            v = self._view(y, o)
            v += row.reshape(v.shape)

    def stiffness(self, u):
        """A u without the boundary conditions; u on the lattice."""
        y = torch.zeros_like(u)
        for t in range(6):
            part = self.K[t] @ self._gather(u, t)
            self._scatter(y, t, part if self.kappa is None else part * self.kappa[t])
        return y

    def mass(self, u):
        y = torch.zeros_like(u)
        for t in range(6):
            self._scatter(y, t, self.M @ self._gather(u, t))
        return y

    def apply(self, u):
        return torch.where(self.inner, self.stiffness(torch.where(self.inner, u, 0.0)), u)

    def diagonal(self):
        y = torch.zeros(self.m, self.m, self.m, dtype=torch.float64, device=DEV)
        one = torch.ones(self.n ** 3, dtype=torch.float64, device=DEV)
        for t in range(6):
            w = one if self.kappa is None else self.kappa[t]
            self._scatter(y, t, torch.diagonal(self.K[t])[:, None] * w)
        return torch.where(self.inner, y, 1.0)

    def load_quadrature(self, f):
        """f: values at the quadrature points, [6 n^3, 27]."""
        xi, w = _gauss_points()
        phi = np.array([[np.prod([p[i] ** e[i] for i in range(3)]) for e in self.expo] for p in xi]) @ self.coef.T
        B = torch.from_numpy(w[:, None] * phi / self.n ** 3).to(DEV)
        b = torch.zeros(self.m, self.m, self.m, dtype=torch.float64, device=DEV)
        f = f.reshape(-1, 6, 27)
        for t in range(6):
            self._scatter(b, t, (f[:, t] @ B).T)
        return torch.where(self.inner, b, 0.0)

    def solve(self, b):
        """Jacobi-preconditioned CG to rounding."""
        dinv = 1 / self.diagonal()
        x, r = torch.zeros_like(b), b.clone()
        z = r * dinv
        p, rz, stop = z.clone(), (r * z).sum(), 1e-14 * b.norm()
        for it in range(6000):
            q = self.apply(p)
            a = rz / (p * q).sum()
            x += a * p
            r -= a * q
            if it % 10 == 9 and r.norm() <= stop:
                break
            z = r * dinv
            rz, old = (r * z).sum(), rz
            p = z + (rz / old) * p
        return x

    def to_lattice(self, v):
        u = torch.empty(self.m ** 3, dtype=torch.float64, device=DEV)
        u[self.order] = v.to(torch.float64)
        return u.reshape(self.m, self.m, self.m)

    def from_lattice(self, u):
        return u.reshape(-1)[self.order]


def _exact_solve(n, k, kappa, f, quad):
    A = _Lattice(n, k, kappa)
    b = A.load_quadrature(f) if quad else torch.where(A.inner, A.mass(A.to_lattice(f)), 0.0)
    return A, A.solve(b)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        out = []
        for p, (n, k) in enumerate(_batch_table(case["problems"], BATCH_SIZES_SEED)):
            if p >= 4:  # the first problems stand for the rest: a plain CG solve of every one takes too long
                out.append(None)
                continue
            A, u = _exact_solve(n, k, _field(_centroids(n), seed, 100 + p), _waves(_coords(n, k), seed, 300 + p), False)
            out.append(A.from_lattice(u))
        return out
    n, k = case["n0"] << case["refine"], case["degree"]
    if kind == "apply":
        A = _Lattice(n, k, _kappa(case, n, seed))
        return A.from_lattice(A.apply(A.to_lattice(_random((k * n + 1) ** 3, seed, 3, DTYPES[case["dtype"]][1]))))
    if kind == "vcycle" or case.get("method") == "fmg_patch" or (k * n + 1) ** 3 > 3_000_000:
        return None  # no closed value, or too large for a plain CG solve
    if kind == "solve":
        A, u = _exact_solve(n, k, _kappa(case, n, seed), _load_input(case, n, seed), case["rhs"] == "quad")
        return A.from_lattice(u)
    kappa = _field(_centroids(n), seed, 7)
    A, u = _exact_solve(n, 1, kappa, torch.ones((n + 1) ** 3, dtype=torch.float64, device=DEV), False)
    diff = u - A.to_lattice(_waves(_coords(n, 1), seed, 13) / 100)
    Md = A.mass(diff)
    lam = A.solve(torch.where(A.inner, -2 * Md, 0.0))
    grad = torch.stack([(A._gather(lam, t) * (A.K[t] @ A._gather(u, t))).sum(0) for t in range(6)], -1)
    return {"J": (diff * Md).sum(), "gradient": grad.reshape(-1)}
