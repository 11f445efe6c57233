"""Where the kernels let their dependents in, read from the sources (no GPU).

A programmatic dependent may be placed as soon as one thread of every CTA has
executed grid_dep_launch.  If its CTA lands on an SM where a CTA of the first
grid has not yet got its tensor memory, it can take the columns and then wait
for that grid, which waits for the columns: both wait for ever.  So a kernel
that allocates tensor memory executes grid_dep_launch only after the barrier
that publishes the allocation, and every kernel only after its own wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2606_00724_gb300", "csrc")
BARRIER = re.compile(r"__syncthreads\(\)|named_sync\(")


def _after_parens(text, i):
    """Index behind the group that opens at text[i]."""
    depth = 0
    for j in range(i, len(text)):
        depth += {"(": 1, ")": -1}.get(text[j], 0)
        if depth == 0:
            return j + 1
    raise ValueError("unbalanced")


def _kernels():
    """(file:name, body without comments) of every kernel that lets dependents in."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        with open(os.path.join(CSRC, f)) as fh:
            text = re.sub(r"//[^\n]*", "", fh.read())
        for m in re.finditer(r"__global__\s+void\s+", text):
            i = m.end()
            if text.startswith("__launch_bounds__", i):
                i = _after_parens(text, text.index("(", i))
            name = re.compile(r"\s*(\w+)").match(text, i).group(1)
            body = text[_after_parens(text, text.index("(", i)):]
            body = body[:body.index("\n}\n")]
            if "grid_dep_launch()" in body:
                yield f"{f}:{name}", body


KERNELS = dict(_kernels())


def test_every_programmatic_kernel_is_looked_at():
    names = {k.split(":")[1] for k in KERNELS}
    assert {"wf_fused_kernel", "wf_gqa_filter_kernel", "tc_attn_kernel", "tc_attn_rows_kernel", "attn_combine_kernel",
            "wf_f32_kernel", "approx_kernel", "approx_stream_kernel"} <= names


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_dependents_come_in_after_the_wait_and_the_allocation(name):
    body = KERNELS[name]
    launch = body.index("grid_dep_launch()")
    assert body.index("grid_dep_wait()") < launch
    if "tmem_alloc(" in body:
        barrier = BARRIER.search(body, body.index("tmem_alloc("))
        assert barrier and barrier.start() < launch
