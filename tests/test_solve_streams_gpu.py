"""The solver's workspace grows on the caller's stream: a context that is used
first by the preconditioner or a narrow solve and then by a wide solve, on
streams that do not wait for the legacy stream, gives the solutions of a
fresh context on the default stream, bit for bit (every reduction of the
solver has a fixed order), and no call touches the legacy stream's memory
operations (read from the source)."""
import os
import re

import numpy as np
import pytest

from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
N, P, NQ = (4, 3, 3), 3, 5
WIDTHS = (4, 36, 132, 260)
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_counters_are_zeroed_on_the_callers_stream():
    with open(os.path.join(ROOT, "paper_2208_07129_gb300", "csrc", "fe_solve.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    body = src[src.index("cudaError_t solver_workspace("):]
    body = body[:body.index("\n}")]
    assert "cudaMemset(" not in body
    assert re.search(r"cudaMemsetAsync\(w\.ticket, 0, .*?, s\);\s*if \(e == cudaSuccess\) e = cudaStreamSynchronize\(s\)",
                     body)


def _context(fe):
    ctx = fe.fe_setup(*N, P, NQ)
    fe.fe_set_potential(ctx, np.full(fe.fe_num_cells(ctx) * NQ ** 3, 2.0))
    return ctx


def _rhs(fe, ctx, nv):
    """A product: zero on the constrained rows, as a right-hand side has to be."""
    x = torch.from_numpy(inputs.random_block(fe.fe_num_dofs(ctx), nv, "normal", nv)).cuda()
    b = torch.empty_like(x)
    fe.fe_apply(ctx, x, b)
    return b


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_growing_solves_on_side_streams(mode):
    from paper_2208_07129_gb300 import build, fe
    build.build()
    want = []
    for nv in WIDTHS:
        ctx = _context(fe)
        b = _rhs(fe, ctx, nv)
        x = torch.zeros_like(b)
        r = fe.fe_solve(ctx, b, x, rtol=1e-10, inner_mode=mode)
        assert r["status"] == fe.FE_OK
        want.append((b, x, r["iterations"]))
        fe.fe_destroy(ctx)
    ctx = _context(fe)
    try:
        n3 = fe.fe_precond_input_size(ctx)
        fe.fe_precond_set_weights(ctx, np.zeros((128, n3)), np.zeros(128), np.zeros((n3, 128)), np.zeros(n3))
        r32 = want[0][0].float()
        z = torch.empty_like(r32)
        torch.cuda.synchronize()
        fe.fe_precond_apply(ctx, r32, z, stream=torch.cuda.Stream())   # grows the workspace for one column
        for b, x, iterations in want:
            s = torch.cuda.Stream()
            y = torch.zeros_like(b)
            torch.cuda.synchronize()
            r = fe.fe_solve(ctx, b, y, rtol=1e-10, inner_mode=mode, stream=s)
            torch.cuda.synchronize()
            assert r["status"] == fe.FE_OK and r["iterations"] == iterations
            assert torch.equal(x, y)
    finally:
        fe.fe_destroy(ctx)
