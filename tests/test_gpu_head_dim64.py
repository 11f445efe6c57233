"""The fused step and the grouped filter for bf16 with head_dim 64, at the
edges of their plans: one query row, ragged lists, clusters of 8 down to 1,
both warpgroups on a unit, no generation rows, token
trim, [B, rows, H, d] strides, blocks of 33 to 64 rows, grouped heads.

Indices and level sets bit-exact against the fp64 oracle on planted inputs.
Outputs: O is rounded to bf16 once, so an element is off by at most half an
ulp (2^-9 of its value, 2^-8 across a power of two) plus the fp32 error of the
sums; P keeps 24 bits and each exponent carries an absolute error of about
|s| 2^-23 with |s| below 150 here, 2e-5 of the largest |V|."""
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


@pytest.mark.parametrize("B,H,group,q,n,L,k,ng,bshd", [
    (1, 3, 1, 1, 2048, 2, 301, 0, False),    # one query row, token trim, no generation rows
    (1, 5, 1, 17, 4104, 3, 512, 7, True),    # ragged n, [B, rows, H, d] strides, an odd unit count
    (2, 16, 1, 32, 8200, 3, 821, 32, True),  # clusters of 4
    (4, 40, 1, 32, 2048, 2, 256, 32, False),  # more units than SMs: one unit a cluster of one CTA, two waves
    (1, 2, 1, 32, 65536, 4, 3277, 64, False),  # lists above 2048: both warpgroups on the unit
    (1, 3, 1, 40, 4104, 3, 513, 5, False),   # blocks of more than 32 rows: the grouped filter
    (1, 2, 4, 32, 4104, 3, 512, 32, True),   # grouped heads
])
def test_step_head_dim64(B, H, group, q, n, L, k, ng, bshd):
    w = synth.Workload("hd64", B, H, 64, n, q, max(ng, 1), L, tuple(wf.wf_default_schedule(n, L, k)), "bf16", "iid",
                       group=group)
    units = [u for u in (0, 1, 7, B * H // 2, B * H - 1) if u < B * H]
    b = synth.make_batch(w, planted=True, device="cuda", cfg="hd64", units=units)
    if bshd:
        b = synth.Batch(*(_bshd(t) for t in (b.Q, b.K, b.V, b.Kg, b.Vg)), b.targets)
    Kg, Vg = (b.Kg, b.Vg) if ng else (None, None)
    run = LibRun(b.Q, b.K, b.V, Kg, Vg, L, w.keep).dwt().step(refresh=False)
    wf.wf_workspace_status(run.ws_step)
    filt = LibRun(b.Q, b.K, b.V, Kg, Vg, L, w.keep).dwt().filter()
    torch.cuda.synchronize()
    assert torch.equal(filt.idx, run.idx) and torch.equal(filt.sets, run.sets)
    for u in units:
        i, h = divmod(u, H)
        Q, K, V = f64(b.Q[i, h * group:(h + 1) * group]), f64(b.K[i, h]), f64(b.V[i, h])
        kg, vg = (f64(Kg[i, h]), f64(Vg[i, h])) if ng else (None, None)
        pyr = oracle.haar_pyramid_spec32(K.astype(np.float32), L, True)
        mu0, sets = oracle.filter_gqa(Q, pyr, K, n, L, np.array(w.keep), want_sets=True)
        got = run.level_sets(u)
        for lev in range(L, -1, -1):
            assert np.array_equal(got[lev], sets[lev]), f"unit {u} scale {lev}"
        assert np.array_equal(run.idx[u].cpu().numpy(), mu0)
        want = oracle.sparse_attn_gqa(Q, K, V, mu0, kg, vg)
        err = np.abs(f64(run.O[i, h * group:(h + 1) * group]) - want)
        bound = 2.0 ** -8 * np.abs(want) + 2e-5 * np.abs(V).max()
        assert (err <= bound).all(), f"unit {u}: {(err - bound).max():.3g} over"
