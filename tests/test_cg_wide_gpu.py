"""Block-PCG over the column counts its vector kernels distinguish (one column
group, a partly filled column tile, several tiles, counts that take the
scalar kernels): every column against the oracle's residual, and a column's
solution does not depend on its neighbours."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["fp64", "fp32"])
@pytest.mark.parametrize("nv", [1, 2, 4, 7, 12, 36, 132, 260])
def test_every_column_solved(nv, mode):
    from paper_2208_07129_gb300 import build, fe
    build.build()
    ctx = fe.fe_setup(3, 2, 2, 3, 5)
    mesh = orc.Mesh(3, 2, 2)
    try:
        V = np.full(mesh.num_cells * 125, 2.0)
        fe.fe_set_potential(ctx, V)
        A = orc.assemble(mesh, 3, 5, Vq=V)
        n = fe.fe_num_dofs(ctx)
        B = inputs.random_block(n, nv, "normal", 5)
        B[orc.constrained_mask(mesh, 3)] = 0.0
        b = torch.from_numpy(B).cuda()
        x = torch.zeros_like(b)
        r = fe.fe_solve(ctx, b, x, rtol=1e-10, inner_mode=mode)
        assert r["status"] == fe.FE_OK and r["converged_columns"] == nv
        res = B - A @ x.cpu().numpy()
        assert np.all(np.linalg.norm(res, axis=0) <= 1.01e-10 * np.linalg.norm(B, axis=0))
    finally:
        fe.fe_destroy(ctx)
