"""The energy x.(A x) of smooth blocks on box meshes: what a solver's step length
and a filter's Rayleigh quotient take from a product.  A constant, one period
and a Gaussian on a periodic box with V = 1, against
    1/2 |grad u_h|^2 + u_h^2
summed over the quadrature points in FP64 as the sum of squares it is, from
the block's own (rounded) values.

Tolerances.  The energy is a sum of squares of values that six passes with N
and N^T and the point operation form.  Each of the seven adds at most 2 u of
relative error that does not average out over the points (the rounding of a
table entry and of a sum that one term dominates): 14 u, taken as 16 u.  FP32:
u = 2^-24.  Double-float: u = 2^-48 (two FP32 significands).  FP64: the host
forms table entries as products of up to 2 (n_q - 1) = 20 rounded factors, so a
pass adds about sqrt(20) u more: 7 (2 + 4.5) u = 46 u, twice that for the
derivative, whose square enters: 92 u.  A stiffness that does not annihilate the constant
exactly adds u |K| / h^2 instead (FP32: 4e-4 for the constant on 12^3 cells, p = 6)."""
import numpy as np
import pytest
from numpy.polynomial import legendre

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp32": 16 * 2.0 ** -24, "df64": 16 * 2.0 ** -48, "fp64": 92 * 2.0 ** -53}
LO, HI = (-1.0, 0.0, 0.5), (0.5, 1.0, 1.5)


@pytest.fixture(scope="module")
def fe():
    from paper_2208_07129_gb300 import build, fe as fe_mod
    build.build()
    fe_mod.lib()
    return fe_mod


def _gll(n):
    c = np.zeros(n)
    c[-1] = 1.0
    inner = np.sort(legendre.legroots(legendre.legder(c)).real) if n > 2 else np.zeros(0)
    for _ in range(3):   # Newton on P'(x), with P'' from Legendre's equation
        d = legendre.legval(inner, legendre.legder(c))
        inner = inner - d * (1 - inner ** 2) / (2 * inner * d - n * (n - 1) * legendre.legval(inner, c))
    x = np.concatenate([[-1.0], inner, [1.0]])
    return x, 2.0 / (n * (n - 1) * legendre.legval(x, c) ** 2)


def _lagrange(x, t):
    """Values and derivatives at t of the Lagrange polynomials on nodes x."""
    diff = x[:, None] - x[None, :] + np.eye(len(x))
    V = np.empty((len(t), len(x)))
    D = np.zeros_like(V)
    for k in range(len(x)):
        others = [j for j in range(len(x)) if j != k]
        V[:, k] = np.prod([(t - x[j]) / diff[k, j] for j in others], axis=0)
        for m in others:
            D[:, k] += np.prod([(t - x[j]) / diff[k, j] for j in others if j != m], axis=0) / diff[k, m]
    return V, D


def _blocks(n, p, gx):
    axes = []
    for d in range(3):
        h = (HI[d] - LO[d]) / n
        axes.append((h * np.arange(n)[:, None] + h * (gx[:-1] + 1) / 2).ravel() / (HI[d] - LO[d]))
    z, y, x = np.meshgrid(axes[2], axes[1], axes[0], indexing="ij")
    period = np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y) * np.sin(2 * np.pi * z + 0.3)
    gauss = np.exp(-((x - 0.5) ** 2 + (y - 0.5) ** 2 + (z - 0.5) ** 2) / (2 * 0.1 ** 2))
    return np.stack([np.ones_like(x), period, gauss], axis=-1).reshape(-1, 3)


def _energy(n, p, nq, gx, qx, qw, X):
    V, D = _lagrange(gx, qx)
    M = n * p
    idx = (np.arange(n)[:, None] * p + np.arange(p + 1)) % M
    h = [(HI[d] - LO[d]) / n for d in range(3)]
    w = np.einsum("a,b,c->abc", qw, qw, qw) * h[0] * h[1] * h[2] / 8
    out = []
    for u in X.T:
        u = u.reshape(M, M, M)
        U = u[idx[:, None, None, :, None, None], idx[None, :, None, None, :, None], idx[None, None, :, None, None, :]]
        U = U.reshape(n ** 3, p + 1, p + 1, p + 1)

        def at(A, B, C):
            t = np.einsum("ck,eijk->eijc", C, U, optimize=True)
            t = np.einsum("bj,eijc->eibc", B, t, optimize=True)
            return np.einsum("ai,eibc->eabc", A, t, optimize=True)

        sq = at(V, V, V) ** 2 + 0.5 * ((2 / h[0]) ** 2 * at(V, V, D) ** 2 + (2 / h[1]) ** 2 * at(V, D, V) ** 2 +
                                       (2 / h[2]) ** 2 * at(D, V, V) ** 2)
        out.append((sq * w).sum())
    return np.array(out)


@pytest.mark.parametrize("p,k,quad", [(p, k, "gauss") for p in range(2, 9) for k in (1, 2, 3)] + [(4, 2, "gll")])
def test_energy_of_smooth_blocks(fe, p, k, quad):
    n, nq = 12 if p <= 4 else 8, p + k
    gx, _ = _gll(p + 1)
    qx, qw = legendre.leggauss(nq) if quad == "gauss" else _gll(nq)
    ctx = fe.fe_setup(n, n, n, p, nq, periodic=True, quad=fe.FE_QUAD_GAUSS if quad == "gauss" else fe.FE_QUAD_GLL, lo=LO, hi=HI)
    try:
        fe.fe_set_potential(ctx, np.ones(fe.fe_num_cells(ctx) * nq ** 3))
        for mode, tol in TOL.items():
            dt = np.float32 if mode == "fp32" else np.float64
            X = _blocks(n, p, gx).astype(dt)
            want = _energy(n, p, nq, gx, qx, qw, X.astype(np.float64))
            fe.fe_set_mode(ctx, mode)
            x = torch.from_numpy(X).cuda()
            y = torch.empty_like(x)
            fe.fe_apply(ctx, x, y)
            got = (x.double() * y.double()).sum(0).cpu().numpy()
            err = np.abs(got - want) / want
            assert np.all(err <= tol), (mode, err, tol)
    finally:
        fe.fe_destroy(ctx)
