"""A batch applied to other blocks from call to call: each call reads and writes
the blocks it was given.  The table of block addresses is staged in pinned
memory, so a call may write it only when the last call's copy has been made."""
import os
import re

import pytest

from paper_2208_07129_gb300 import inputs

torch = pytest.importorskip("torch")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_table_is_written_after_the_last_copy():
    with open(os.path.join(ROOT, "paper_2208_07129_gb300", "csrc", "fe_batch.cu")) as f:
        src = re.sub(r"//[^\n]*", "", f.read())
    body = src[src.index("fe_status fe_batch_apply("):]
    body = body[:body.index("\n}")]
    wait, write, copy = (body.index(k) for k in ("cudaStreamSynchronize(s)", "h_ptrs[2 * i] =", "cudaMemcpyAsync("))
    assert wait < write < copy


@pytest.mark.gpu
@pytest.mark.parametrize("mode", ["fp64", "fp32"])
def test_blocks_change_from_call_to_call(mode):
    from paper_2208_07129_gb300 import build, fe
    build.build()
    ctxs = [fe.fe_setup(2, 2, 2, 3, 5), fe.fe_setup(3, 2, 2, 4, 6)]
    nv = [8, 5]
    dt = torch.float32 if mode == "fp32" else torch.float64
    try:
        X = [[torch.from_numpy(inputs.random_block(fe.fe_num_dofs(c), v, "normal", 7 * k + i)).to("cuda", dt)
              for i, (c, v) in enumerate(zip(ctxs, nv))] for k in range(20)]
        Y = [[torch.full_like(x, float("nan")) for x in xs] for xs in X]
        batch = fe.fe_batch_create(ctxs, nv, mode=mode, autotune=False)
        torch.cuda.synchronize()
        for xs, ys in zip(X, Y):
            fe.fe_batch_apply(batch, xs, ys)
        torch.cuda.synchronize()
        fe.fe_batch_destroy(batch)
        for xs, ys in zip(X, Y):
            for c, x, y in zip(ctxs, xs, ys):
                fe.fe_set_mode(c, mode)
                want = torch.empty_like(x)
                fe.fe_apply(c, x, want)
                assert torch.equal(y, want)
    finally:
        for c in ctxs:
            fe.fe_destroy(c)
