"""The preconditioner's application over the sizes its task loop distinguishes:
one to three output chunks, more and fewer tasks than SMs, ragged column
blocks; against the FP64 oracle with the kernel's bfloat16 roundings.

Tolerances as in the inference test: one bfloat16 rounding of a hidden value
may fall the other way after an FP32 sum (2^-9 of it), 2e-3 over the block."""
import numpy as np
import pytest

from oracle import mlp_oracle as mo
from oracle import oracle as orc
from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,n,nv,periodic", [(1, (6, 5, 4), 1, False), (2, (3, 3, 3), 129, True), (4, (2, 3, 2), 128, False),
                                             (5, (3, 2, 2), 257, False), (6, (2, 2, 3), 127, True),
                                             (3, (7, 6, 8), 300, False)])
def test_application_matches_oracle(p, n, nv, periodic):
    from paper_2208_07129_gb300 import build, fe
    build.build()
    ctx = fe.fe_setup(*n, p, p + 2, periodic=periodic)
    mesh = orc.Mesh(*n, periodic=periodic)
    try:
        fe.fe_set_potential(ctx, np.ones(mesh.num_cells * (p + 2) ** 3))   # no zero diagonal on a periodic box
        dofs, n3 = fe.fe_num_dofs(ctx), (p + 1) ** 3
        rng = np.random.default_rng(p)
        W = (rng.normal(0, 0.2, (128, n3)).astype(np.float32), rng.normal(0, 0.1, 128).astype(np.float32),
             rng.normal(0, 0.2, (n3, 128)).astype(np.float32), rng.normal(0, 0.1, n3).astype(np.float32))
        fe.fe_precond_set_weights(ctx, *W)
        r = inputs.random_block(dofs, nv, "normal", 3).astype(np.float32)   # boundary rows too: z = D^-1 r there
        Z = torch.full((dofs, nv), float("nan"), dtype=torch.float32, device="cuda")
        fe.fe_precond_apply(ctx, torch.from_numpy(r).cuda(), Z)
        torch.cuda.synchronize()
        assert fe.fe_last_device_status(ctx) == fe.FE_OK
        d = torch.empty(dofs, dtype=torch.float64, device="cuda")
        fe.fe_diagonal(ctx, d)
        dinv = (1.0 / d.cpu().numpy()).astype(np.float32).astype(np.float64)
        ref = mo.precond(mesh, p, r.astype(np.float64), dinv, *[w.astype(np.float64) for w in W], bf16=True)
        got = Z.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(got - ref) <= 2e-3 * np.linalg.norm(ref)
        assert np.abs(got - ref).max() < 2e-2 * np.abs(ref).max()
    finally:
        fe.fe_destroy(ctx)
