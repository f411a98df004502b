"""Batches whose largest tile asks for nearly 48 KB of shared memory: the kernel's
own static shared memory comes on top, and the launch needs the attribute for
larger requests although the tile alone does not (p = 7, four vectors, FP64: 47,360
bytes beside the staged tables)."""
import pytest

from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp64", "df64", "fp32"])
@pytest.mark.parametrize("p", [5, 7])
@pytest.mark.parametrize("nv", [4, 8, 16])
def test_tiles_around_48_kilobytes(mode, p, nv):
    from paper_2208_07129_gb300 import build, fe
    build.build()
    ctxs = [fe.fe_setup(2, 2, 2, p, p + 2), fe.fe_setup(2, 1, 2, 3, 5)]
    try:
        dt = torch.float32 if mode == "fp32" else torch.float64
        X = [torch.from_numpy(inputs.random_block(fe.fe_num_dofs(c), nv, "normal", i)).to("cuda", dt)
             for i, c in enumerate(ctxs)]
        Y = [torch.full_like(x, float("nan")) for x in X]
        batch = fe.fe_batch_create(ctxs, [nv] * 2, mode=mode, autotune=False)
        fe.fe_batch_apply(batch, X, Y)
        torch.cuda.synchronize()
        fe.fe_batch_destroy(batch)
        for c, x, y in zip(ctxs, X, Y):
            fe.fe_set_mode(c, mode)
            want = torch.empty_like(x)
            fe.fe_apply(c, x, want)
            assert torch.equal(y, want)
    finally:
        for c in ctxs:
            fe.fe_destroy(c)
