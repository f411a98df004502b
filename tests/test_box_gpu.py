"""The box-cell kernel (fe_box.cuh: separable stiffness, one matrix per direction)
over every compiled (p, n_q): against the oracle on anisotropic boxes, through
the colour-ordered launches and the small-mesh path, and against the trilinear
kernel on the same box given by its vertices.

Tolerances: those of the modes (FP64 and double-float 1e-12, FP32 2e-6: the
bounds of chained contractions of length <= 11 in the mode's arithmetic,
which the separable form does not lengthen)."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "df64": 1e-12, "fp32": 2e-6}
PAIRS = [(p, p + k) for p in range(1, 9) for k in (1, 2, 3)]
BOX = dict(lo=(-1.0, 0.0, 0.5), hi=(0.5, 0.4, 1.5))   # cell sizes 0.5, 0.2, 0.25 on 3 x 2 x 4 cells


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


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("p,nq", PAIRS)
def test_box_kernel_every_size(fe, p, nq, periodic):
    n = (3, 2, 4)
    ctx = fe.fe_setup(*n, p, nq, periodic=periodic, **BOX)
    mesh = orc.Mesh(*n, periodic=periodic, **BOX)
    try:
        fe.fe_set_potential(ctx, inputs.coulomb_potential(fe.fe_quadrature_points(ctx)))
        V = inputs.coulomb_potential(orc.quad_points(mesh, p, nq))
        # 133 columns: no small-mesh path in any mode; a ragged last tile
        X = inputs.random_block(fe.fe_num_dofs(ctx), 133, "normal", p)
        for mode in ("fp64", "df64", "fp32"):
            Xr = X.astype(np.float32).astype(np.float64) if mode == "fp32" else X
            ref = orc.apply(mesh, p, nq, Xr[:, :9], Vq=V)
            Y = _apply(fe, ctx, X, mode)
            got = Y[:, :9].double().cpu().numpy()
            scale = np.abs(ref).max()
            assert np.linalg.norm(got - ref) <= TOL[mode] * np.linalg.norm(ref), mode
            assert np.abs(got - ref).max() <= TOL[mode] * scale, mode
            assert torch.isfinite(Y).all()
            # the small-mesh path and other widths give the same columns bit for bit
            for w in (1, 9, 50):
                assert torch.equal(_apply(fe, ctx, np.ascontiguousarray(X[:, :w]), mode), Y[:, :w]), (mode, w)
    finally:
        fe.fe_destroy(ctx)


@pytest.mark.parametrize("mode", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("p,nq", [(1, 2), (3, 5), (4, 7), (6, 8), (8, 9)])
def test_box_equals_trilinear_kernel(fe, p, nq, mode):
    """The same box with and without vertices: two kernels, one operator."""
    n = (3, 2, 4)
    z, y, x = np.meshgrid(*(np.linspace(BOX["lo"][d], BOX["hi"][d], n[d] + 1) for d in (2, 1, 0)), indexing="ij")
    verts = np.stack([x, y, z], axis=-1).reshape(-1, 3)
    a, b = fe.fe_setup(*n, p, nq, **BOX), fe.fe_setup(*n, p, nq, vertices=verts)
    try:
        for c in (a, b):
            fe.fe_set_potential(c, inputs.coulomb_potential(fe.fe_quadrature_points(c)))
        X = inputs.random_block(fe.fe_num_dofs(a), 70, "uniform", 3)
        Ya, Yb = _apply(fe, a, X, mode), _apply(fe, b, X, mode)
        assert (Ya - Yb).norm() <= TOL[mode] * Yb.norm()
    finally:
        fe.fe_destroy(a)
        fe.fe_destroy(b)


@pytest.mark.parametrize("mode", ["fp64", "df64", "fp32"])
def test_batch_of_different_aspects(fe, mode):
    """Problems of one degree whose cells differ in shape do not share tables."""
    ctxs = [fe.fe_setup(4, 4, 4, 4, 6), fe.fe_setup(4, 2, 5, 4, 6), fe.fe_setup(3, 3, 3, 4, 6, hi=(2.0, 2.0, 2.0)),
            fe.fe_setup(2, 3, 2, 5, 7, **BOX), fe.fe_setup(3, 3, 3, 4, 6, hi=(2.0, 1.0, 1.0))]
    nv = [20, 7, 33, 12, 5]
    try:
        dt = torch.float32 if mode == "fp32" else torch.float64
        X = [torch.from_numpy(inputs.random_block(fe.fe_num_dofs(c), v, "normal", i)).to("cuda", dt)
             for i, (c, v) in enumerate(zip(ctxs, nv))]
        Y = [torch.full_like(x, float("nan")) for x in X]
        batch = fe.fe_batch_create(ctxs, nv, mode=mode, autotune=False)
        fe.fe_batch_apply(batch, X, Y)
        torch.cuda.synchronize()
        assert fe.fe_batch_stats(batch, len(ctxs))["device_status"] == 0
        fe.fe_batch_destroy(batch)
        for c, x, y in zip(ctxs, X, Y):
            fe.fe_set_mode(c, mode)
            want = torch.empty_like(x)
            fe.fe_apply(c, x, want)
            assert torch.equal(y, want)
    finally:
        for c in ctxs:
            fe.fe_destroy(c)
