"""Tensor memory and overlapping launches, read from the sources (no GPU): a
kernel that allocates tensor memory with a blocking allocation and lets the
next launch start must keep a CTA of the next launch from taking the memory
its own CTAs still wait for.  Either the allocation has returned before the
next launch may start, or shared memory keeps two CTAs off one SM; the
preconditioner, whose tables shrink with the degree, does both."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_07129_gb300", "csrc")


def _source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_every_allocating_kernel_is_listed():
    users = sorted(n for n in os.listdir(CSRC) if "tcgen05.alloc" in _source(n))
    assert users == ["fe_learn.cu", "fe_tc_kernel.cuh"]


def test_preconditioner_allocates_before_the_next_launch_may_start():
    src = _source("fe_learn.cu")
    kernel = src[src.index("mlp_precond_kernel("):]
    alloc, start = kernel.index("tcgen05.alloc"), kernel.index("let_next_launch_start()")
    assert alloc < kernel.index("__syncthreads()", alloc) < start


def test_one_cta_per_sm():
    learn, tc = _source("fe_learn.cu"), _source("fe_apply_tc.cu")
    assert re.search(r"static_assert\(2 \* mlp_smem_request\(16\) > kSmSharedBytes", learn)
    assert "kSmSharedBytes = 228 * 1024" in learn
    launch = learn[learn.index("fe_status precond_apply_f32("):]
    assert re.search(r"smem = mlp_smem_request\(", launch) and "mlp_smem_bytes(" not in launch
    assert re.search(r"static_assert\(2 \* \(SH::SMEM_BYTES \+ 1024\) > 228 \* 1024", tc)
