"""Products on unaligned blocks, inside a captured graph, and on two streams of
one context: the launches overlap and small meshes use a scratch, and neither
may show in the results."""
import numpy as np
import pytest

from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SMALL, LARGE = (3, 3, 2), (5, 4, 4)      # below and above the small-mesh limit at p = 6


@pytest.fixture(scope="module")
def fe():
    from paper_2208_07129_gb300 import build, fe as fe_mod
    build.build()
    fe_mod.lib()
    return fe_mod


def _context(fe, n, bent, mode):
    ctx = fe.fe_setup(*n, 6, 8, vertices=inputs.perturbed_vertices(*n, seed=1) if bent else None)
    fe.fe_set_potential(ctx, inputs.coulomb_potential(fe.fe_quadrature_points(ctx)))
    fe.fe_set_mode(ctx, mode)
    return ctx


def _block(fe, ctx, nv, mode, seed):
    dt = torch.float32 if mode == "fp32" else torch.float64
    return torch.from_numpy(inputs.random_block(fe.fe_num_dofs(ctx), nv, "normal", seed)).to("cuda", dt)


@pytest.mark.parametrize("mode", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("bent", [False, True])
@pytest.mark.parametrize("n", [SMALL, LARGE])
def test_unaligned_blocks(fe, n, bent, mode):
    ctx = _context(fe, n, bent, mode)
    try:
        X = _block(fe, ctx, 12, mode, 1)
        Y = torch.empty_like(X)
        fe.fe_apply(ctx, X, Y)
        for dx, dy in ((1, 0), (0, 1), (1, 1)):
            x = torch.empty(X.numel() + 1, dtype=X.dtype, device="cuda")[dx:dx + X.numel()].view_as(X)
            y = torch.full((X.numel() + 1,), float("nan"), dtype=X.dtype, device="cuda")[dy:dy + X.numel()].view_as(X)
            x.copy_(X)
            fe.fe_apply(ctx, x, y)
            assert torch.equal(y, Y)
    finally:
        fe.fe_destroy(ctx)


@pytest.mark.parametrize("mode", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("bent", [False, True])
@pytest.mark.parametrize("n", [SMALL, LARGE])
def test_captured_product(fe, n, bent, mode):
    ctx = _context(fe, n, bent, mode)
    try:
        X, Y = _block(fe, ctx, 10, mode, 2), None
        Y = torch.empty_like(X)
        fe.fe_apply(ctx, X, Y)      # kernel attributes are set before the capture
        Z = torch.empty_like(X)
        s = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=s):
            fe.fe_apply(ctx, X, Y)
            fe.fe_apply(ctx, Y, Z)
        for seed in (3, 4):
            X.copy_(_block(fe, ctx, 10, mode, seed))
            Y.fill_(float("nan"))
            Z.fill_(float("nan"))
            g.replay()
            torch.cuda.synchronize()
            y, z = torch.empty_like(X), torch.empty_like(X)
            fe.fe_apply(ctx, X, y)
            fe.fe_apply(ctx, y, z)
            assert torch.equal(Y, y) and torch.equal(Z, z)
    finally:
        fe.fe_destroy(ctx)


def test_double_float_products_on_two_streams(fe):
    """Small double-float products of one context need no order between streams."""
    ctx = _context(fe, SMALL, False, "df64")
    try:
        X = [_block(fe, ctx, 16, "df64", 5 + k) for k in range(2)]
        want = []
        for x in X:
            want.append(torch.empty_like(x))
            fe.fe_apply(ctx, x, want[-1])
        torch.cuda.synchronize()
        streams = [torch.cuda.Stream() for _ in range(2)]
        Y = [[torch.empty_like(x) for _ in range(50)] for x in X]
        torch.cuda.synchronize()
        for r in range(50):
            for k in range(2):
                fe.fe_apply(ctx, X[k], Y[k][r], stream=streams[k])
        torch.cuda.synchronize()
        for k in range(2):
            assert all(torch.equal(y, want[k]) for y in Y[k])
    finally:
        fe.fe_destroy(ctx)


def test_captured_preconditioner(fe):
    ctx = fe.fe_setup(3, 2, 2, 4, 6)
    try:
        n3 = fe.fe_precond_input_size(ctx)
        rng = np.random.default_rng(0)
        fe.fe_precond_set_weights(ctx, rng.normal(size=(128, n3)), np.zeros(128), 0.01 * rng.normal(size=(n3, 128)),
                                  np.zeros(n3))
        R = torch.from_numpy(inputs.random_block(fe.fe_num_dofs(ctx), 20, "normal", 1)).to("cuda", torch.float32)
        Z, W = torch.empty_like(R), torch.empty_like(R)
        fe.fe_precond_apply(ctx, R, Z)
        s, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=s):
            fe.fe_precond_apply(ctx, R, W)
        W.fill_(float("nan"))
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(W, Z)
    finally:
        fe.fe_destroy(ctx)
