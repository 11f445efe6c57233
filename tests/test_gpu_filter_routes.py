"""Which kernels wf_filter takes, at the edges of each route: the fused kernel
without its attention (bf16, head_dim 128, at most 32 query rows, one query
head a key head), the grouped filter kernel (grouped heads, blocks of 33 to 64
rows), and the kernels per scale past those kernels' 8192 candidates a scale.  Indices and
level sets bit-exact against the fp64 oracle on planted inputs, which have a
margin at every Top-K boundary; also for [B, rows, H, d] strides and without
level sets."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from helpers import LibRun, f64
from paper_2606_00724_gb300 import synth, wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)


def _bshd(t):
    return t.transpose(1, 2).contiguous().transpose(1, 2)


@pytest.mark.parametrize("B,H,group,q,n,L,k,bshd", [
    (1, 3, 1, 1, 2048, 1, 301, False),    # one query row, one scale, an odd k (token trim)
    (1, 1, 1, 32, 256, 3, 8, True),       # one unit, fewer candidates than one tile
    (2, 3, 1, 32, 4104, 3, 512, True),    # ragged n, [B, rows, H, d] strides
    (1, 2, 1, 17, 16384, 1, 4096, False),  # 8192 candidates: the largest list of the fused kernel
    (1, 1, 1, 17, 16640, 1, 4096, False),  # 8320 candidates: the kernels per scale
    (1, 2, 4, 32, 4104, 3, 513, True),    # grouped heads, ragged n, token trim
    (1, 3, 1, 33, 4104, 3, 513, True),    # the smallest block above the fused kernel's: two chunks of query columns
    (1, 2, 1, 64, 8192, 4, 820, False),   # the largest block
    (1, 1, 4, 64, 2048, 2, 301, False),   # grouped heads with blocks of 64: 256 stacked rows
    (1, 1, 3, 5, 2048, 2, 256, False),    # grouped heads that fit one chunk
])
def test_filter_route(B, H, group, q, n, L, k, bshd):
    w = synth.Workload("filter_route", B, H, 128, n, q, 1, L, tuple(wf.wf_default_schedule(n, L, k)), "bf16", "iid",
                       group=group)
    b = synth.make_batch(w, planted=True, device="cuda", cfg="route")
    if bshd:
        b = dataclasses.replace(b, Q=_bshd(b.Q), K=_bshd(b.K), V=_bshd(b.V))
    run = LibRun(b.Q, b.K, b.V, None, None, L, w.keep).dwt().filter()
    bare = LibRun(b.Q, b.K, b.V, None, None, L, w.keep, want_sets=False).dwt().filter()
    torch.cuda.synchronize()
    assert torch.equal(bare.idx, run.idx)
    for u in range(w.units):
        i, h = divmod(u, H)
        K = f64(b.K[i, h])
        pyr = oracle.haar_pyramid_spec32(K.astype(np.float32), L, True)
        mu0, sets = oracle.filter_gqa(f64(b.Q[i, h * group:(h + 1) * group]), pyr, K, n, L, np.array(w.keep),
                                      want_sets=True)
        assert np.array_equal(run.idx[u].cpu().numpy(), mu0), f"unit {u}"
        got = run.level_sets(u)
        for lev in range(L, -1, -1):
            assert np.array_equal(got[lev], sets[lev]), f"unit {u} scale {lev}"


@pytest.mark.parametrize("B,H,group,q,n,L,k", [
    (1, 20, 7, 32, 16384, 3, 2048),  # clusters of 6 or 7: three tiles a slice, every one kept in the ring
    (3, 30, 4, 32, 16384, 3, 2048),  # one CTA a cluster: 16 tiles a scale, one M tile
    (3, 30, 8, 32, 16384, 3, 2048),  # the same with two M tiles (three ring stages): 13 tiles streamed again
    (5, 40, 1, 48, 4096, 2, 512),    # more units than SMs, a ragged chunk of query rows
])
def test_grouped_filter_streams_again(B, H, group, q, n, L, k):
    # The grouped filter's second pass multiplies the tiles that are still in
    # the ring and streams the others again.
    w = synth.Workload("grouped_filter", B, H, 128, n, q, 1, L, tuple(wf.wf_default_schedule(n, L, k)), "bf16", "iid",
                       group=group)
    units = [0, B * H // 2, B * H - 1]
    b = synth.make_batch(w, planted=True, device="cuda", cfg="grouped", units=units)
    run = LibRun(b.Q, b.K, b.V, None, None, L, w.keep).dwt().filter()
    torch.cuda.synchronize()
    for u in units:
        got = run.level_sets(u)
        for lev in range(L, -1, -1):
            assert np.array_equal(got[lev], b.targets[u][lev].cpu().numpy()), f"unit {u} scale {lev}"


@pytest.mark.parametrize("B,H,group,q,n,L,k", [
    (4, 40, 8, 4, 16384, 1, 2048),   # 160 units: a last wave of 8, a long list: the kernels per scale
    (4, 40, 8, 4, 4096, 1, 512),     # a short one: the grouped kernel
    (2, 40, 2, 3, 16384, 1, 2049),   # half a wave, token trim
    (5, 61, 4, 5, 8192, 2, 819),     # three waves, nearly full
])
def test_grouped_filter_line(B, H, group, q, n, L, k):
    # Up to 32 stacked rows and one CTA a unit: where the plan prefers the
    # kernels per scale, and beside that line; the filter and the step.
    w = synth.Workload("grouped_line", B, H, 128, n, q, 1, L, tuple(wf.wf_default_schedule(n, L, k)), "bf16", "iid",
                       group=group)
    units = [0, B * H // 2, B * H - 1]
    b = synth.make_batch(w, planted=True, device="cuda", cfg="line", units=units)
    run = LibRun(b.Q, b.K, b.V, None, None, L, w.keep).dwt().filter()
    step = LibRun(b.Q, b.K, b.V, None, None, L, w.keep).dwt().step(refresh=False)
    wf.wf_workspace_status(step.ws_step)
    torch.cuda.synchronize()
    for u in units:
        got, again = run.level_sets(u), step.level_sets(u)
        for lev in range(L, -1, -1):
            assert np.array_equal(got[lev], b.targets[u][lev].cpu().numpy()), f"unit {u} scale {lev}"
            assert np.array_equal(again[lev], got[lev]), f"unit {u} scale {lev} of the step"
