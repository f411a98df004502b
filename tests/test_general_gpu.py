"""The trilinear cell kernel (fe_general.cuh) over every compiled (p, n_q)
against the oracle on a perturbed mesh: colour-ordered launches, the
small-mesh path, ragged widths.

Tolerances: those of the modes (FP64 and double-float 1e-12, FP32 2e-6: the
bounds of chained contractions of length <= 11 in the mode's arithmetic)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "df64": 1e-12, "fp32": 2e-6}
PAIRS = [(p, p + k) for p in range(1, 9) for k in (1, 2, 3)]


@pytest.fixture(scope="module")
def fe():
    from paper_2208_07129_gb300 import build, fe as fe_mod
    build.build()
    fe_mod.lib()
    return fe_mod


def _apply(fe, ctx, X, mode):
    fe.fe_set_mode(ctx, mode)
    x = torch.from_numpy(X).to("cuda", torch.float32 if mode == "fp32" else torch.float64).contiguous()
    y = torch.full_like(x, float("nan"))
    fe.fe_apply(ctx, x, y)
    torch.cuda.synchronize()
    return y


@pytest.mark.parametrize("p,nq", PAIRS)
def test_trilinear_kernel_every_size(fe, p, nq):
    n = (3, 2, 3)
    verts = inputs.perturbed_vertices(*n, seed=40 + p)
    ctx = fe.fe_setup(*n, p, nq, vertices=verts)
    mesh = orc.Mesh(*n, vertices=verts)
    try:
        fe.fe_set_potential(ctx, inputs.coulomb_potential(fe.fe_quadrature_points(ctx)))
        V = inputs.coulomb_potential(orc.quad_points(mesh, p, nq))
        X = inputs.random_block(fe.fe_num_dofs(ctx), 133, "normal", p)   # above the small-mesh path in any mode
        for mode in ("fp64", "df64", "fp32"):
            Xr = X.astype(np.float32).astype(np.float64) if mode == "fp32" else X
            ref = orc.apply(mesh, p, nq, Xr[:, :9], Vq=V)
            Y = _apply(fe, ctx, X, mode)
            got = Y[:, :9].double().cpu().numpy()
            assert np.linalg.norm(got - ref) <= TOL[mode] * np.linalg.norm(ref), mode
            assert np.abs(got - ref).max() <= TOL[mode] * np.abs(ref).max(), mode
            assert torch.isfinite(Y).all()
            for w in (1, 9, 50):
                assert torch.equal(_apply(fe, ctx, np.ascontiguousarray(X[:, :w]), mode), Y[:, :w]), (mode, w)
    finally:
        fe.fe_destroy(ctx)
