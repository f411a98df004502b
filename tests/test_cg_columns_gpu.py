"""Block-PCG's column sums: joined in FP64 over the threads of a CTA (read from
the source; no result shows the difference of a few bits, since each thread's
own FP32 sum is a few FP32 ulps off), and independent from column to column:
the columns of a block on the vector kernels have the solutions they have in a
narrower block, after about as many iterations as on the scalar kernels."""
import os
import re

import numpy as np
import pytest

from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_thread_sums_are_joined_in_fp64():
    with open(os.path.join(ROOT, "paper_2208_07129_gb300", "csrc", "fe_solve.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    acc = src[src.index("struct ColAcc<float> {"):]
    assert "double value() const" in acc[:acc.index("};")]
    finish = src[src.index("void wide_finish("):]
    finish = finish[:finish.index("__threadfence")]
    assert "__shared__ double red[" in finish and "ff" not in re.findall(r"\w+", finish)


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_columns_do_not_depend_on_their_neighbours(mode):
    """Tolerance: both residuals are at most 1e-10 |b|, so the solutions lie at
    most 2e-10 |b| / (smallest eigenvalue of A) apart.  The iteration count may
    move by the four between two checks per refinement step, and by a tenth
    with rounding."""
    from paper_2208_07129_gb300 import build, fe
    build.build()
    ctx = fe.fe_setup(4, 3, 3, 3, 5)
    try:
        fe.fe_set_potential(ctx, np.full(fe.fe_num_cells(ctx) * 125, 2.0))
        n = fe.fe_num_dofs(ctx)
        X0 = torch.from_numpy(inputs.random_block(n, 36, "normal", 3)).cuda()
        B = torch.empty_like(X0)
        fe.fe_apply(ctx, X0, B)

        def solve(cols):
            b = B[:, cols].contiguous()
            x = torch.zeros_like(b)
            info = fe.fe_solve(ctx, b, x, rtol=1e-10, inner_mode=mode)
            assert info["status"] == fe.FE_OK
            return x, info

        wide, info = solve(list(range(36)))
        some, _ = solve(list(range(8, 20)))
        narrow = [solve(list(range(7 * k, min(36, 7 * k + 7)))) for k in range(6)]
        A = torch.empty(n, n, dtype=torch.float64, device="cuda")
        fe.fe_apply(ctx, torch.eye(n, dtype=torch.float64, device="cuda"), A)
        free = A.abs().sum(0) > 0
        low = torch.linalg.eigvalsh(A[free][:, free])[0].item()
        bound = 2e-10 * B.norm(dim=0) / low
        assert low > 0 and (bound < 1e-4 * X0[free].norm(dim=0)).all()
        assert ((wide[:, 8:20] - some).norm(dim=0) <= bound[8:20]).all()
        assert ((wide - torch.cat([x for x, _ in narrow], dim=1)).norm(dim=0) <= bound).all()
        most = max(i["iterations"] for _, i in narrow)
        steps = max(i["outer_iterations"] for _, i in narrow + [(None, info)])
        assert info["iterations"] <= 1.1 * most + 4 * (1 + steps)
    finally:
        fe.fe_destroy(ctx)
