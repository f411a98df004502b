"""Batches of meshes whose cells differ in shape: one kernel per degree, whatever
the aspects; every result is fe_apply's bit for bit, and the batch costs about
what the same work with one aspect costs (a kernel per aspect cost 2.5 times
as much with 24 of them)."""
import pytest

from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fe():
    from paper_2208_07129_gb300 import build, fe as fe_mod
    build.build()
    fe_mod.lib()
    return fe_mod


def _dtype(mode):
    return torch.float32 if mode == "fp32" else torch.float64


@pytest.mark.parametrize("mode", ["df64", "fp32", "fp64"])
def test_every_degree_with_and_without_one_aspect(fe, mode):
    """Degrees 3..8: each with two aspects, and once more with one."""
    for aspects in (2, 1):
        ctxs = [fe.fe_setup(2 + i % 2, 2, 3, p, p + 2, periodic=bool(i),
                            hi=(1.0 + i % 2, 1.0, 1.5 * (1.0 + 0.3 * (i % aspects))))
                for p in range(3, 9) for i in range(2)]
        try:
            nv = [3 + 5 * i for i in range(len(ctxs))]
            for c in ctxs:
                fe.fe_set_potential(c, inputs.coulomb_potential(fe.fe_quadrature_points(c)))
            X = [torch.from_numpy(inputs.random_block(fe.fe_num_dofs(c), v, "normal", i)).to("cuda", _dtype(mode))
                 for i, (c, v) in enumerate(zip(ctxs, nv))]
            Y = [torch.full_like(x, float("nan")) for x in X]
            batch = fe.fe_batch_create(ctxs, nv, mode=mode, autotune=False)
            for _ in range(2):
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


def _batch_ms(fe, mode, aspects, count=24):
    ctxs = [fe.fe_setup(8, 8, 8, 4, 6, hi=(1.0, 1.0, 1.0 + 0.05 * (i % aspects))) for i in range(count)]
    try:
        X = [torch.ones(fe.fe_num_dofs(c), 32, device="cuda", dtype=_dtype(mode)) for c in ctxs]
        Y = [torch.empty_like(x) for x in X]
        batch = fe.fe_batch_create(ctxs, [32] * count, mode=mode, autotune=False)
        times = []
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            fe.fe_batch_apply(batch, X, Y)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        fe.fe_batch_destroy(batch)
        return min(times)
    finally:
        for c in ctxs:
            fe.fe_destroy(c)


@pytest.mark.parametrize("mode", ["df64", "fp32"])
def test_many_aspects_cost_what_one_does(fe, mode):
    assert _batch_ms(fe, mode, 24) <= 1.4 * _batch_ms(fe, mode, 1)
