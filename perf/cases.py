"""Timed cases of the library: what programs built on it call, through its Python binding.

A case is a dict of plain values.  ``op`` names the call:

* ``apply``    Y = A X (``fe_apply``) on a structured mesh, box or trilinear cells, in one arithmetic mode;
* ``refined``  the same product on a one-level refined mesh with hanging nodes;
* ``filter``   the Chebyshev filter of the eigen layer (``fe_chebyshev_filter``);
* ``solve``    block-PCG with Jacobi to a relative residual of 1e-12 (``fe_solve``);
* ``batch``    uneven problems in one persistent launch (``fe_batch_apply``);
* ``precond``  one application of the learned cell-patch preconditioner (``fe_precond_apply``).

``exact`` evaluates the same definitions in 64 bits with torch and numpy alone.
"""
import itertools
import math

import numpy as np
import torch

from paper_2208_07129_gb300 import fe

GAUSSIANS = 8
FILTER_DEGREE = 40
SOLVE_RTOL = 1e-12
HIDDEN = 128
MU = 0.5


def listed():
    return [
        # a small operator applied many times (an inner step of a user's own loop): launches and latency count
        dict(name="fp64_small", op="apply", mode="fp64", nx=4, ny=4, nz=4, p=4, nq=6, nv=8, periodic=False, bent=False),
        # the benchmark's product: a periodic electronic-structure box, FP64
        dict(name="fp64_periodic", op="apply", mode="fp64", nx=32, ny=32, nz=32, p=6, nq=8, nv=64, periodic=True,
             bent=False),
        # a deformed mesh at the highest degree, many vectors, FP64
        dict(name="fp64_trilinear", op="apply", mode="fp64", nx=16, ny=16, nz=16, p=8, nq=10, nv=256, periodic=False,
             bent=True),
        # the benchmark's product with FP64 data in double-float arithmetic
        dict(name="df64_periodic", op="apply", mode="df64", nx=32, ny=32, nz=32, p=6, nq=8, nv=64, periodic=True,
             bent=False),
        # an adaptively refined mesh with hanging nodes
        dict(name="df64_refined", op="refined", mode="df64", nx=14, ny=14, nz=14, r0=3, r1=11, p=6, nq=8, nv=64),
        # the operator of the 128-right-hand-side solve's inner iterations
        dict(name="fp32_box", op="apply", mode="fp32", nx=24, ny=24, nz=24, p=6, nq=8, nv=128, periodic=False,
             bent=False),
        # a deformed mesh of ordinary size, odd cell counts and a block width that fills no tile
        dict(name="fp32_trilinear_odd", op="apply", mode="fp32", nx=13, ny=9, nz=11, p=5, nq=7, nv=50, periodic=False,
             bent=True),
        # reduced-precision products on the tensor cores
        dict(name="bf16_periodic", op="apply", mode="bf16", nx=32, ny=32, nz=32, p=6, nq=8, nv=64, periodic=True,
             bent=False),
        # one filter pass of the subspace iteration for 100 eigenpairs
        dict(name="fp64_filter", op="filter", mode="fp64", nx=8, ny=8, nz=8, p=6, nq=8, nv=128),
        # a mixed-precision solve: FP32 inner iterations, FP64 refinement
        dict(name="mixed_solve", op="solve", mode="fp32", nx=12, ny=12, nz=12, p=6, nq=8, nv=32),
        # uneven problems together: n, degree, vectors
        dict(name="fp64_batch", op="batch", mode="fp64", problems="12,6,96 7,4,45 9,8,23 16,3,130 5,7,11 20,5,8"),
        # the learned preconditioner inside the 128-right-hand-side solve
        dict(name="precond", op="precond", mode="fp32", nx=24, ny=24, nz=24, p=6, nq=8, nv=128),
    ]


# rough passes per second of DoF x vector, used by draw() to keep a drawn case below the largest listed one
RATE = {"fp64": 2e9, "df64": 6e9, "fp32": 2e10, "tf32": 2e10, "bf16": 3e10, "bf16s": 3e10, "tf32x3": 1e10}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, lo, hi):
    n = _log(rng, lo, hi)
    return [max(2, n + rng.randint(-n // 4, n // 4)) for _ in range(3)]


def draw(rng):
    op = rng.choice(["apply"] * 6 + ["refined", "filter", "solve", "batch", "precond"])
    while True:
        nv = _log(rng, 1, 256)
        if op == "apply":
            mode = rng.choice(["fp64", "fp64", "df64", "df64", "fp32", "fp32", "tf32", "bf16", "bf16s", "tf32x3"])
            p = rng.randint(2, 8)
            if mode in ("tf32", "bf16", "bf16s", "tf32x3"):
                p = rng.randint(3, 6)
            nq = p + rng.choice([2, 2, 2, 1])
            n = _mesh(rng, 2, 32)
            c = dict(op=op, mode=mode, nx=n[0], ny=n[1], nz=n[2], p=p, nq=nq, nv=nv, periodic=rng.random() < 0.4,
                     bent=False)
            c["bent"] = not c["periodic"] and rng.random() < 0.4
            cost = _dofs(c) * nv / RATE[mode]
        elif op == "refined":
            mode = rng.choice(["fp64", "df64", "fp32"])
            p = rng.randint(2, 6)
            n = rng.randint(3, 12)
            r0 = rng.randint(0, n // 2)
            c = dict(op=op, mode=mode, nx=n, ny=n, nz=n, r0=r0, r1=rng.randint(r0 + 1, n), p=p, nq=p + 2, nv=nv)
            cost = _cells(c) * p ** 3 * nv / RATE[mode]
        elif op == "filter":
            mode = rng.choice(["fp64", "df64", "fp32"])
            p = rng.randint(2, 7)
            n = _mesh(rng, 2, 12)
            c = dict(op=op, mode=mode, nx=n[0], ny=n[1], nz=n[2], p=p, nq=p + 2, nv=nv)
            cost = FILTER_DEGREE * _dofs(c) * nv / RATE[mode]
        elif op == "solve":
            mode = rng.choice(["fp32", "fp32", "fp64", "df64"])
            p = rng.randint(2, 6)
            n = _mesh(rng, 3, 12)
            nv = min(nv, 64)
            c = dict(op=op, mode=mode, nx=n[0], ny=n[1], nz=n[2], p=p, nq=p + 2, nv=nv)
            cost = _iterations(c) * (_dofs(c) * nv / min(RATE[mode], 6e9) + 1e-4)
        elif op == "batch":
            mode = rng.choice(["fp64", "df64", "fp32"])
            sets = [(_log(rng, 4, 20), rng.randint(3, 8), _log(rng, 8, 256)) for _ in range(rng.randint(2, 8))]
            c = dict(op=op, mode=mode, problems=" ".join("%d,%d,%d" % s for s in sets))
            cost = sum((n * p) ** 3 * v for n, p, v in sets) / RATE[mode]
        else:
            p = rng.randint(2, 6)
            n = _mesh(rng, 2, 24)
            c = dict(op=op, mode="fp32", nx=n[0], ny=n[1], nz=n[2], p=p, nq=p + 2, nv=nv)
            cost = _dofs(c) * max(nv, 128) / 2e10
        if cost <= 0.15:
            return c


# ---------------------------------------------------------------- sizes and work


def _dofs(c):
    add = 0 if c.get("periodic") else 1
    return (c["nx"] * c["p"] + add) * (c["ny"] * c["p"] + add) * (c["nz"] * c["p"] + add)


def _cells(c):
    n = c["nx"] * c["ny"] * c["nz"]
    return n + 7 * (c["r1"] - c["r0"]) ** 3 if c["op"] == "refined" else n


def _iterations(c):
    """Jacobi-PCG iterations to SOLVE_RTOL, as they come out for these operators."""
    return 8 * max(c["nx"], c["ny"], c["nz"]) * c["p"]


def _bytes(mode):
    return 8 if mode in ("fp64", "df64") else 2 if mode == "bf16s" else 4


def _product(dofs, cells, np_, nq, nv, elem, bent):
    """One product: X read, Y written, the coefficients read; the sum-factorised operations of a cell (box cells have a
    separable stiffness: one symmetric matrix per direction at the points)."""
    f = 4 * (np_ ** 3 * nq + np_ ** 2 * nq ** 2 + np_ * nq ** 3) + (12 * nq ** 4 + 16 * nq ** 3 if bent else
                                                                    6 * nq ** 4 + 4 * nq ** 3)
    coef = cells * nq ** 3 * (7 if bent else 1) * max(elem, 4)
    return 2 * dofs * nv * elem + coef, cells * nv * f


def work(case):
    c, e = case, _bytes(case["mode"])
    if c["op"] == "batch":
        b = f = 0
        for n, p, v in _problems(c):
            x, y = _product((n * p) ** 3, n ** 3, p + 1, p + 2, v, e, False)
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    dofs, cells = _dofs(c), _cells(c)
    if c["op"] == "refined":
        r = c["r1"] - c["r0"]
        dofs += (2 * r * c["p"]) ** 3 - (r * c["p"]) ** 3
    b, f = _product(dofs, cells, c["p"] + 1, c["nq"], c["nv"], e, c.get("bent", False))
    if c["op"] == "filter":
        return {"bytes": FILTER_DEGREE * b, "flops": FILTER_DEGREE * f}
    if c["op"] == "solve":   # per iteration the product, and x, r, p read and written
        k = _iterations(c)
        return {"bytes": k * (b + 6 * dofs * c["nv"] * e), "flops": k * f}
    if c["op"] == "precond":
        return {"bytes": 2 * dofs * c["nv"] * 4, "flops": cells * c["nv"] * 4 * HIDDEN * (c["p"] + 1) ** 3}
    return {"bytes": b, "flops": f}


def _problems(c):
    return [tuple(int(x) for x in s.split(",")) for s in c["problems"].split()]


# ---------------------------------------------------------------- inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _potential(seed, periodic, xyz, shift):
    """V at (..., 3) points (torch, 64 bits): minus a sum of Gaussians, plus `shift`."""
    rng = np.random.default_rng(1000 + seed)
    centres, widths = rng.uniform(0.0, 1.0, (GAUSSIANS, 3)), rng.uniform(0.05, 0.2, GAUSSIANS)
    out = torch.full(xyz.shape[:-1], float(shift), dtype=torch.float64, device=xyz.device)
    for c, s in zip(centres, widths):
        d = xyz - torch.tensor(c, dtype=torch.float64, device=xyz.device)
        if periodic:
            d -= torch.round(d)
        out -= torch.exp(-(d * d).sum(-1) / (2.0 * s * s))
    return out


def _shift(c):
    """The solves shift the operator so that it is positive definite."""
    return float(GAUSSIANS) if c["op"] == "solve" else 0.0


def _vertices(c, seed):
    """Vertices of the unit cube's grid, the interior ones moved by up to a fifth of the cell size."""
    n = (c["nx"], c["ny"], c["nz"])
    rng = np.random.default_rng(2000 + seed)
    z, y, x = np.meshgrid(np.arange(n[2] + 1), np.arange(n[1] + 1), np.arange(n[0] + 1), indexing="ij")
    h = 1.0 / np.array(n, dtype=np.float64)
    v = np.stack([x * h[0], y * h[1], z * h[2]], axis=-1).reshape(-1, 3)
    inner = ((x > 0) & (x < n[0]) & (y > 0) & (y < n[1]) & (z > 0) & (z < n[2])).reshape(-1)
    v[inner] += rng.uniform(-0.2, 0.2, v.shape)[inner] * h
    return np.ascontiguousarray(v)


def _block(dofs, nv, mode, seed):
    """The multivector of a case: normal values in the element type of the mode."""
    g = torch.Generator(device=_device()).manual_seed(seed)
    dtype = {8: torch.float64, 4: torch.float32, 2: torch.bfloat16}[_bytes(mode)]
    if dtype == torch.bfloat16:
        return torch.randn(dofs, nv, generator=g, device=_device(), dtype=torch.float32).to(dtype)
    return torch.randn(dofs, nv, generator=g, device=_device(), dtype=dtype)


def _boundary(c):
    """Mask of the Dirichlet nodes of a structured box."""
    n = [c[k] * c["p"] + 1 for k in ("nx", "ny", "nz")]
    m = torch.zeros(n[2], n[1], n[0], dtype=torch.bool, device=_device())
    m[0] = m[-1] = m[:, 0] = m[:, -1] = m[:, :, 0] = m[:, :, -1] = True
    return m.reshape(-1)


def _weights(c, seed):
    n3 = (c["p"] + 1) ** 3
    rng = np.random.default_rng(3000 + seed)
    f = np.float32
    return (rng.normal(0, 1, (HIDDEN, n3)).astype(f), rng.normal(0, 0.1, HIDDEN).astype(f),
            rng.normal(0, 0.01, (n3, HIDDEN)).astype(f), rng.normal(0, 0.01, n3).astype(f))


def _bounds(c):
    """(lambda_min, lambda_u, lambda_max) of the filter: the box Laplacian's spectrum bounds the operator's."""
    pi = math.pi
    low = sorted(MU * pi * pi * (i * i + j * j + k * k) for i, j, k in itertools.product(range(1, 13), repeat=3))
    top = 0.0
    x, w = _gll(c["p"] + 1)
    d = _lagrange(x, _gauss(c["p"] + 1)[0])[1]
    k1 = (d * _gauss(c["p"] + 1)[1][:, None]).T @ d
    for n in (c["nx"], c["ny"], c["nz"]):
        size = n * c["p"] + 1
        k, m = np.zeros((size, size)), np.zeros(size)
        for e in range(n):
            at = slice(e * c["p"], e * c["p"] + c["p"] + 1)
            k[at, at] += k1 * 2 * n
            m[at] += w / (2 * n)
        top += MU * np.linalg.eigvalsh(k / np.sqrt(m[:, None] * m[None, :]))[-1]
    want = low[min(len(low) - 1, max(c["nv"], 4))]
    return low[0] - 2.0, min(want, 0.5 * top), 1.01 * top


# ---------------------------------------------------------------- the library


class Operator:
    """A context of the library, released with this object."""

    def __init__(self, c, seed):
        if c["op"] == "refined":
            r0, r1 = (c["r0"],) * 3, (c["r1"],) * 3
            self.ctx = fe.fe_setup_refined(c["nx"], c["ny"], c["nz"], c["p"], c["nq"], r0, r1, mu=MU)
        else:
            self.ctx = fe.fe_setup(c["nx"], c["ny"], c["nz"], c["p"], c["nq"], periodic=c.get("periodic", False),
                                   vertices=_vertices(c, seed) if c.get("bent") else None, mu=MU)
        xyz = torch.from_numpy(fe.fe_quadrature_points(self.ctx)).to(_device())
        v = _potential(seed, c.get("periodic", False), xyz, _shift(c))
        fe.fe_set_potential(self.ctx, v.cpu().numpy())
        if c["op"] not in ("solve", "batch", "precond"):
            fe.fe_set_mode(self.ctx, c["mode"])

    def __del__(self):
        if getattr(self, "ctx", None):
            fe.fe_destroy(self.ctx)


class Batch:
    """A batch over operators, released before them."""

    def __init__(self, ops, nv, mode):
        self.ops = ops
        self.handle = fe.fe_batch_create([o.ctx for o in ops], nv, mode=mode)

    def __del__(self):
        if getattr(self, "handle", None):
            fe.fe_batch_destroy(self.handle)


def _part(c, k):
    n, p, v = _problems(c)[k]
    return dict(op="batch", mode=c["mode"], nx=n, ny=n, nz=n, p=p, nq=p + 2, nv=v, periodic=True)


def prepare(case, seed):
    c = case
    s = {"op": c["op"], "mode": c["mode"]}
    if c["op"] == "batch":
        parts = [_part(c, k) for k in range(len(_problems(c)))]
        ops = [Operator(q, seed + k) for k, q in enumerate(parts)]
        s["batch"] = Batch(ops, [q["nv"] for q in parts], c["mode"])
        s["X"] = [_block(_dofs(q), q["nv"], c["mode"], seed + k) for k, q in enumerate(parts)]
        s["Y"] = [torch.empty_like(x) for x in s["X"]]
        return s
    op = s["operator"] = Operator(c, seed)
    if c["op"] == "solve":
        s["B"] = _block(_dofs(c), c["nv"], "fp64", seed)
        s["B"][_boundary(c)] = 0.0
        s["X"] = torch.zeros_like(s["B"])
        return s
    s["X"] = _block(fe.fe_num_dofs(op.ctx), c["nv"], c["mode"], seed)
    s["Y"] = torch.empty_like(s["X"])
    if c["op"] == "filter":
        s["U"] = torch.empty_like(s["X"])
        s["bounds"] = _bounds(c)
    if c["op"] == "precond":
        fe.fe_precond_set_weights(op.ctx, *_weights(c, seed))
    return s


def run(state):
    s = state
    if s["op"] == "batch":
        fe.fe_batch_apply(s["batch"].handle, s["X"], s["Y"])
        return s["Y"]
    ctx = s["operator"].ctx
    if s["op"] == "solve":
        s["X"].zero_()
        fe.fe_solve(ctx, s["B"], s["X"], rtol=SOLVE_RTOL, inner_mode=s["mode"])
        return s["X"]
    if s["op"] == "filter":
        s["U"].copy_(s["X"])
        fe.fe_chebyshev_filter(ctx, s["U"], s["Y"], FILTER_DEGREE, *s["bounds"])
        return s["U"]
    if s["op"] == "precond":
        fe.fe_precond_apply(ctx, s["X"], s["Y"])
        return s["Y"]
    fe.fe_apply(ctx, s["X"], s["Y"])
    return s["Y"]


# ---------------------------------------------------------------- 64-bit reference


def _gauss(n):
    return np.polynomial.legendre.leggauss(n)


def _gll(n):
    """Gauss-Lobatto-Legendre nodes and weights on [-1, 1]."""
    leg = np.polynomial.legendre.Legendre.basis(n - 1)
    x = np.concatenate([[-1.0], np.sort(leg.deriv().roots().real), [1.0]])
    for _ in range(2):   # Newton on (1 - x^2) P'
        f, d = leg.deriv()(x[1:-1]), leg.deriv(2)(x[1:-1])
        x[1:-1] -= f / d
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (n * (n - 1) * leg(x) ** 2)


def _lagrange(nodes, at):
    """Values and derivatives (points x nodes) of the Lagrange basis."""
    n = len(nodes)
    val, der = np.ones((len(at), n)), np.zeros((len(at), n))
    for i in range(n):
        others = [j for j in range(n) if j != i]
        for j in others:
            val[:, i] *= (at - nodes[j]) / (nodes[i] - nodes[j])
        for k in others:
            t = np.full(len(at), 1.0 / (nodes[i] - nodes[k]))
            for j in others:
                if j != k:
                    t *= (at - nodes[j]) / (nodes[i] - nodes[j])
            der[:, i] += t
    return val, der


def _along(m, u, axis):
    """m applied to one of the node axes (1, 2, 3 = z, y, x) of u (cells, z, y, x, vectors)."""
    shape = list(u.shape)
    left, right = int(np.prod(shape[:axis])), int(np.prod(shape[axis + 1:]))
    v = torch.matmul(m, u.reshape(left, shape[axis], right))
    return v.reshape(shape[:axis] + [m.shape[0]] + shape[axis + 1:])


class Exact:
    """The operator of a case in 64 bits: cells, their nodes, the metric and the potential."""

    def __init__(self, c, seed):
        self.c, self.dev = c, _device()
        p, nq = c["p"], c["nq"]
        self.g, self.wg = _gll(p + 1)
        self.q, self.wq = _gauss(nq)
        val, der = _lagrange(self.g, self.q)
        self.N, self.B = self.t(val), self.t(der)
        if c["op"] == "refined":
            self.refined_nodes()
        else:
            self.box_nodes()
        self.geometry(seed)
        c3 = 1.0 / torch.bincount(self.nodes.reshape(-1), minlength=self.n).double()
        self.share = c3[self.nodes]

    def t(self, a):
        return torch.as_tensor(a, dtype=torch.float64, device=self.dev)

    def box_nodes(self):
        c, p = self.c, self.c["p"]
        axes = []
        for k in ("nx", "ny", "nz"):
            i = np.arange(c[k])[:, None] * p + np.arange(p + 1)
            axes.append(i % (c[k] * p) if c.get("periodic") else i)
        size = [c[k] * p + (0 if c.get("periodic") else 1) for k in ("nx", "ny", "nz")]
        gx, gy, gz = axes
        nodes = (gx[None, None, :, None, None, :] + size[0] * (gy[None, :, None, None, :, None] +
                                                               size[1] * gz[:, None, None, :, None, None]))
        self.nodes = torch.from_numpy(nodes.reshape(-1, (p + 1) ** 3)).to(self.dev)
        self.n = size[0] * size[1] * size[2]
        self.fixed = torch.zeros(self.n, dtype=torch.bool, device=self.dev) if c.get("periodic") else _boundary(c)
        z, y, x = np.meshgrid(np.arange(c["nz"]), np.arange(c["ny"]), np.arange(c["nx"]), indexing="ij")
        h = np.array([1.0 / c["nx"], 1.0 / c["ny"], 1.0 / c["nz"]])
        self.lo = np.stack([x, y, z], axis=-1).reshape(-1, 3) * h
        self.h = np.broadcast_to(h, self.lo.shape)
        self.slaves = None

    def refined_nodes(self):
        """Cells in order (a refined cell replaced by its children), nodes identified and numbered by position, and the
        hanging nodes with the weights of the coarse neighbour's interpolant."""
        c, p = self.c, self.c["p"]
        n, r0, r1 = c["nx"], c["r0"], c["r1"]
        cells = []
        for cz, cy, cx in itertools.product(range(n), repeat=3):
            if all(r0 <= i < r1 for i in (cx, cy, cz)):
                cells += [(1, 2 * cx + (k & 1), 2 * cy + (k >> 1 & 1), 2 * cz + (k >> 2)) for k in range(8)]
            else:
                cells.append((0, cx, cy, cz))
        cells = np.array(cells)
        level, index = cells[:, 0], cells[:, 1:]
        size = np.where(level == 1, 2.0, 4.0)            # in quarters of a coarse cell
        pos = index[:, :, None] * size[:, None, None] + (1.0 + self.g) * (size / 2)[:, None, None]   # cells, xyz, i
        _, first, rank = np.unique(np.round(pos * 1e8).astype(np.int64), return_index=True, return_inverse=True)
        every, rank = pos.reshape(-1)[first], rank.reshape(pos.shape)
        m = len(every)
        key = (rank[:, 0, None, None, :] + m * (rank[:, 1, None, :, None] + m * rank[:, 2, :, None, None]))
        code, nodes = np.unique(key.reshape(-1), return_inverse=True)
        nodes = nodes.reshape(len(cells), -1)
        self.n = len(code)
        where = every[np.stack([code % m, code // m % m, code // (m * m)], axis=-1)]
        fixed = (np.abs(where) < 1e-6).any(1) | (np.abs(where - 4 * n) < 1e-6).any(1)
        coarse = np.zeros(self.n, dtype=bool)
        coarse[nodes[level == 0].reshape(-1)] = True
        owner_of = np.full((n, n, n), -1)                # coarse cells by (z, y, x)
        at = np.nonzero(level == 0)[0]
        owner_of[index[at, 2], index[at, 1], index[at, 0]] = at
        owner = np.full(self.n, -1)
        for up in itertools.product((0, 1), repeat=3):
            i = np.where(up, np.floor(where / 4 + 1e-7), np.ceil(where / 4 - 1e-7) - 1).astype(int)
            ok = ((i >= 0) & (i < n)).all(1) & (owner < 0)
            i = np.clip(i, 0, n - 1)
            owner = np.where(ok, owner_of[i[:, 2], i[:, 1], i[:, 0]], owner)
        hang = np.nonzero((owner >= 0) & ~coarse & ~fixed)[0]
        local = where[hang] / 2 - 2.0 * index[owner[hang]] - 1.0
        w = [_lagrange(self.g, local[:, k])[0] for k in range(3)]
        self.slaves = torch.from_numpy(hang).to(self.dev)
        self.masters = torch.from_numpy(nodes[owner[hang]]).to(self.dev)
        self.w = self.t((w[2][:, :, None, None] * w[1][:, None, :, None] * w[0][:, None, None, :]).reshape(len(hang), -1))
        self.nodes = torch.from_numpy(nodes).to(self.dev)
        self.fixed = torch.from_numpy(fixed).to(self.dev)
        H = 1.0 / n
        self.h = np.broadcast_to((size * H / 4)[:, None], index.shape)
        self.lo = index * self.h

    def geometry(self, seed):
        c, nq, E = self.c, self.c["nq"], len(self.nodes)
        w3 = self.t(self.wq[:, None, None] * self.wq[None, :, None] * self.wq[None, None, :])
        r = self.t((self.q + 1) / 2)
        if c.get("bent"):
            v = self.t(_vertices(c, seed)).reshape(c["nz"] + 1, c["ny"] + 1, c["nx"] + 1, 3)
            xyz, J = 0, [0, 0, 0]
            for dz, dy, dx in itertools.product((0, 1), repeat=3):
                corner = v[dz:dz + c["nz"], dy:dy + c["ny"], dx:dx + c["nx"]].reshape(E, 1, 1, 1, 3)
                f = [(r if d else 1 - r) for d in (dx, dy, dz)]
                s = [0.5 if d else -0.5 for d in (dx, dy, dz)]
                fx, fy, fz = f[0][None, None, :], f[1][None, :, None], f[2][:, None, None]
                one = torch.ones(nq, nq, nq, dtype=torch.float64, device=self.dev)
                xyz = xyz + corner * (fx * fy * fz)[None, ..., None]
                J[0] = J[0] + corner * (one * s[0] * fy * fz)[None, ..., None]
                J[1] = J[1] + corner * (one * s[1] * fx * fz)[None, ..., None]
                J[2] = J[2] + corner * (one * s[2] * fx * fy)[None, ..., None]
            cross = [torch.linalg.cross(J[(k + 1) % 3], J[(k + 2) % 3], dim=-1) for k in range(3)]
            det = (J[0] * cross[0]).sum(-1)              # rows of det J J^-1 are the cross products
            scale = MU * w3 / det
            self.G = {(i, j): ((cross[i] * cross[j]).sum(-1) * scale)[..., None] for i in range(3) for j in range(3)}
        else:
            h, lo = self.t(self.h.copy()), self.t(self.lo)
            full = torch.zeros(E, nq, nq, nq, dtype=torch.float64, device=self.dev)
            xyz = torch.stack([full + lo[:, 0, None, None, None] + h[:, 0, None, None, None] * r[None, None, None, :],
                               full + lo[:, 1, None, None, None] + h[:, 1, None, None, None] * r[None, None, :, None],
                               full + lo[:, 2, None, None, None] + h[:, 2, None, None, None] * r[None, :, None, None]], -1)
            det = (h.prod(1) / 8)[:, None, None, None]
            self.G = {(i, i): (MU * det * (4.0 / h[:, i] ** 2)[:, None, None, None] * w3)[..., None] for i in range(3)}
        self.C = (_potential(seed, c.get("periodic", False), xyz, _shift(c)) * det * w3)[..., None]

    def cells_product(self, u):
        """A^(e) on (cells, z, y, x, vectors)."""
        ux, dx = _along(self.N, u, 3), _along(self.B, u, 3)
        uxy = _along(self.N, ux, 2)
        d = [_along(self.N, _along(self.N, dx, 2), 1), _along(self.N, _along(self.B, ux, 2), 1), _along(self.B, uxy, 1)]
        val = self.C * _along(self.N, uxy, 1)
        d = [sum(self.G[i, j] * d[j] for j in range(3) if (i, j) in self.G) for i in range(3)]
        Nt, Bt = self.N.T.contiguous(), self.B.T.contiguous()
        vxy = _along(Nt, val, 1) + _along(Bt, d[2], 1)
        vx = _along(Nt, vxy, 2) + _along(Bt, _along(Nt, d[1], 1), 2)
        return _along(Nt, vx, 3) + _along(Bt, _along(Nt, _along(Nt, d[0], 1), 2), 3)

    def __call__(self, X):
        """A X, constraints included, on a 64-bit block."""
        k = self.c["p"] + 1
        Y = torch.empty_like(X)
        E = len(self.nodes)
        width = max(1, min(X.shape[1], int(1.5e8 / (E * self.c["nq"] ** 3)) or 1))
        for a in range(0, X.shape[1], width):
            x = X[:, a:a + width].clone()
            x[self.fixed] = 0
            if self.slaves is not None:
                for i in range(0, len(self.slaves), 8192):
                    j = slice(i, i + 8192)
                    x[self.slaves[j]] = torch.einsum("sm,smv->sv", self.w[j], x[self.masters[j]])
            y = torch.zeros_like(x)
            step = max(1, int(1.5e8 / (self.c["nq"] ** 3 * x.shape[1])))
            for e in range(0, E, step):
                at = self.nodes[e:e + step]
                sub = self.part(e, e + step)
                out = sub.cells_product(x[at].reshape(len(at), k, k, k, -1))
                y.index_add_(0, at.reshape(-1), out.reshape(at.numel(), -1))
            if self.slaves is not None:
                for i in range(0, len(self.slaves), 8192):
                    j = slice(i, i + 8192)
                    t = self.w[j][..., None] * y[self.slaves[j]][:, None, :]
                    y.index_add_(0, self.masters[j].reshape(-1), t.reshape(-1, t.shape[-1]))
                y[self.slaves] = 0
            y[self.fixed] = 0
            Y[:, a:a + width] = y
        return Y

    def part(self, a, b):
        if a == 0 and b >= len(self.nodes):
            return self
        s = object.__new__(Exact)
        s.N, s.B, s.C = self.N, self.B, self.C[a:b]
        s.G = {k: g[a:b] for k, g in self.G.items()}
        return s

    def diagonal(self):
        """diag(A) of a box mesh, 1 on the Dirichlet nodes."""
        N2, B2 = (self.N ** 2).T.contiguous(), (self.B ** 2).T.contiguous()
        at = lambda x, mz, my, mx: _along(mx, _along(my, _along(mz, x, 1), 2), 3)  # noqa: E731
        d = at(self.C, N2, N2, N2)
        for i, m in ((0, (N2, N2, B2)), (1, (N2, B2, N2)), (2, (B2, N2, N2))):
            d = d + at(self.G[i, i].expand_as(self.C).contiguous(), *m)
        out = torch.zeros(self.n, dtype=torch.float64, device=self.dev)
        out.index_add_(0, self.nodes.reshape(-1), d.reshape(-1))
        out[self.fixed] = 1
        return out[:, None]

    def mass(self):
        """Diagonal of the overlap matrix by the rule on the element's own nodes, 1 on the Dirichlet nodes."""
        w = self.t(self.wg[:, None, None] * self.wg[None, :, None] * self.wg[None, None, :]).reshape(-1)
        det = self.t(self.h.copy()).prod(1) / 8
        out = torch.zeros(self.n, dtype=torch.float64, device=self.dev)
        out.index_add_(0, self.nodes.reshape(-1), (det[:, None] * w).reshape(-1))
        out[self.fixed] = 1
        return out[:, None]


def exact(case, seed):
    c = case
    if c["op"] == "batch":
        parts = [_part(c, k) for k in range(len(_problems(c)))]
        return [Exact(q, seed + k)(_block(_dofs(q), q["nv"], c["mode"], seed + k).double())
                for k, q in enumerate(parts)]
    A = Exact(c, seed)
    X = _block(A.n, c["nv"], "fp64" if c["op"] == "solve" else c["mode"], seed).double()
    if c["op"] in ("apply", "refined"):
        return A(X)
    if c["op"] == "filter":
        return _exact_filter(c, A, X)
    if c["op"] == "solve":
        X[A.fixed] = 0
        return _exact_solve(c, A, X)
    return _exact_precond(c, A, X, seed)


def _exact_filter(c, A, X):
    low, cut, top = _bounds(c)
    root = A.mass().rsqrt()
    H = lambda u: root * A(root * u)  # noqa: E731
    e, mid = (top - cut) / 2, (top + cut) / 2
    free = ~A.fixed[:, None]
    X = X * free
    s = s1 = e / (low - mid)
    old, new = X, (H(X) - mid * X) * (s / e)
    for _ in range(FILTER_DEGREE - 1):
        s2 = 1.0 / (2.0 / s1 - s)
        old, new = new, (H(new) - mid * new) * (2 * s2 / e) - (s * s2) * old
        s = s2
    return new


def _exact_solve(c, A, B):
    d = 1.0 / A.diagonal()
    norm = B.norm(dim=0)
    x, r = torch.zeros_like(B), B.clone()
    z = d * r
    p, rz = z.clone(), (r * z).sum(0)
    for k in range(40 * _iterations(c)):
        q = A(p)
        a = torch.where(rz > 0, rz / (p * q).sum(0), torch.zeros_like(rz))
        x += a * p
        r -= a * q
        if k % 10 == 9:
            if float((r.norm(dim=0) / norm).max()) < 1e-14:
                break
        z = d * r
        new = (r * z).sum(0)
        p = z + torch.where(rz > 0, new / rz, torch.zeros_like(rz)) * p
        rz = new
    return x


def _exact_precond(c, A, R, seed):
    w1, b1, w2, b2 = (A.t(w) for w in _weights(c, seed))
    Z = R / A.diagonal()
    x = R.clone()
    x[A.fixed] = 0
    step = max(1, int(1e8 / (A.nodes.shape[1] * R.shape[1])))
    for e in range(0, len(A.nodes), step):
        at = A.nodes[e:e + step]
        u = x[at].permute(0, 2, 1)                       # cells, vectors, nodes
        s = u.norm(dim=-1, keepdim=True)
        y = torch.relu(u @ w1.T / torch.where(s > 0, s, 1.0) + b1) @ w2.T + b2
        y = (y * s * A.share[e:e + step][:, None, :]).permute(0, 2, 1)
        y = y * ~A.fixed[at][..., None]
        Z.index_add_(0, at.reshape(-1), y.reshape(at.numel(), -1))
    return Z
