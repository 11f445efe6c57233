"""The one-launch fp32 step and filter at the edges of its plan: one query
row, blocks of 33 to 64 rows, ragged lists, clusters of 8 down to 1, one tile
buffer or two, slices of several tiles, no generation rows, token trim,
[B, rows, H, d] strides, and the kernels per scale past 8192 candidates.
Indices and level sets bit-exact against the fp64 oracle on planted inputs,
outputs within the fp32 bound (max-abs 1e-5)."""
import numpy as np
import pytest
import torch

import oracle
from helpers import LibRun, assert_close_out, f64
from paper_2606_00724_gb300 import synth, wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)


def _bshd(t):
    return t.transpose(1, 2).contiguous().transpose(1, 2)


@pytest.mark.parametrize("B,H,d,q,n,L,k,ng,bshd", [
    (1, 3, 64, 1, 2048, 2, 301, 0, False),      # one query row, token trim, no generation rows
    (1, 1, 128, 32, 64, 3, 8, 5, True),         # fewer rows than CTAs in the cluster
    (1, 5, 128, 17, 4104, 3, 512, 7, True),     # ragged n, [B, rows, H, d] strides
    (2, 3, 64, 33, 4104, 3, 513, 32, False),    # the smallest block of the 64-row kernels
    (1, 2, 128, 64, 8192, 4, 820, 64, False),   # the largest block
    (2, 40, 64, 32, 2048, 2, 256, 32, False),   # one CTA a cluster: slices of several tiles
    (3, 50, 128, 32, 2048, 2, 205, 3, False),   # the same with one tile buffer
    (1, 1, 128, 32, 16384, 1, 4096, 1, False),  # 8192 candidates, the largest list
    (1, 1, 64, 32, 16640, 1, 4096, 1, False),   # 8320: the kernels per scale
])
def test_step_f32(B, H, d, q, n, L, k, ng, bshd):
    w = synth.Workload("f32", B, H, d, n, q, max(ng, 1), L, tuple(wf.wf_default_schedule(n, L, k)), "f32", "iid")
    units = [u for u in (0, 1, 7, B * H // 2, B * H - 1) if u < B * H]
    b = synth.make_batch(w, planted=True, device="cuda", cfg="f32", units=units)
    if bshd:
        b = synth.Batch(*(_bshd(t) for t in (b.Q, b.K, b.V, b.Kg, b.Vg)), b.targets)
    Kg, Vg = (b.Kg, b.Vg) if ng else (None, None)
    run = LibRun(b.Q, b.K, b.V, Kg, Vg, L, w.keep).dwt().step(refresh=False)
    filt = LibRun(b.Q, b.K, b.V, Kg, Vg, L, w.keep, want_sets=False).dwt().filter()
    torch.cuda.synchronize()
    assert torch.equal(filt.idx, run.idx)
    for u in units:
        i, h = divmod(u, H)
        Q, K, V = f64(b.Q[i, h]), f64(b.K[i, h]), f64(b.V[i, h])
        kg, vg = (f64(Kg[i, h]), f64(Vg[i, h])) if ng else (None, None)
        pyr = oracle.haar_pyramid_spec32(K.astype(np.float32), L, False)
        mu0, sets = oracle.filter(Q, pyr, K, n, L, np.array(w.keep), want_sets=True)
        got = run.level_sets(u)
        for lev in range(L, -1, -1):
            assert np.array_equal(got[lev], sets[lev]), f"unit {u} scale {lev}"
        assert np.array_equal(run.idx[u].cpu().numpy(), mu0)
        assert_close_out(f64(run.O[i, h]), oracle.sparse_attn(Q, K, V, mu0, kg, vg), torch.float32)


@pytest.mark.parametrize("H,d,q,n,L,k,ng,bshd", [
    (153, 128, 5, 2048, 1, 205, 7, True),    # filter and attention leave the one launch
    (153, 64, 17, 2048, 2, 205, 0, False),   # the attention alone does
    (38, 64, 1, 8192, 1, 819, 32, False),    # one wave would do, its slices do not fit the row buffer
    (100, 64, 32, 4096, 2, 411, 3, True),    # two waves of the one launch, token trim
])
def test_step_f32_routes(H, d, q, n, L, k, ng, bshd):
    """Small query blocks where the one launch takes several waves or tiles:
    the routes that the plan's costs choose between."""
    w = synth.Workload("f32", 1, H, d, n, q, max(ng, 1), L, tuple(wf.wf_default_schedule(n, L, k)), "f32", "iid")
    units = [0, H // 2, H - 1]
    b = synth.make_batch(w, planted=True, device="cuda", cfg="f32", units=units)
    if bshd:
        b = synth.Batch(*(_bshd(t) for t in (b.Q, b.K, b.V, b.Kg, b.Vg)), b.targets)
    Kg, Vg = (b.Kg, b.Vg) if ng else (None, None)
    run = LibRun(b.Q, b.K, b.V, Kg, Vg, L, w.keep).dwt().step(refresh=False)
    filt = LibRun(b.Q, b.K, b.V, Kg, Vg, L, w.keep).dwt().filter()
    torch.cuda.synchronize()
    for u in units:
        got, alone = run.level_sets(u), filt.level_sets(u)
        for lev in range(L, -1, -1):
            want = b.targets[u][lev].cpu().numpy()
            assert np.array_equal(np.asarray(got[lev]), want), f"unit {u} scale {lev}"
            assert np.array_equal(np.asarray(alone[lev]), want), f"unit {u} scale {lev}, the filter alone"
        Q, K, V = f64(b.Q[0, u]), f64(b.K[0, u]), f64(b.V[0, u])
        kg, vg = (f64(Kg[0, u]), f64(Vg[0, u])) if ng else (None, None)
        assert_close_out(f64(run.O[0, u]), oracle.sparse_attn(Q, K, V, run.idx[u].cpu().numpy(), kg, vg), torch.float32)


@pytest.mark.parametrize("d,q,n,k,amp", [(128, 8, 4096, 410, 1.0), (128, 32, 8192, 819, 2.0), (64, 17, 4096, 410, 2.0)])
def test_split_attention_as_accurate_as_one_launch(d, q, n, k, amp):
    """A step that leaves the one launch attends on the split kernel.  Both sum
    a logit in two chains of d / 2 products, and the logits' rounding dominates
    the output's, so their rms errors against fp64 agree within a fifth (a
    single chain of d has 1.4 times the error)."""
    H, L, ng = 32, 2, 32
    g = torch.Generator().manual_seed(k + d)
    rn = lambda rows, a=1.0: a * torch.randn(1, H, rows, d, generator=g).cuda()
    Q, K, V, Kg, Vg = rn(q, amp), rn(n), rn(n), rn(ng), rn(ng)
    run = LibRun(Q, K, V, Kg, Vg, L, wf.wf_default_schedule(n, L, k)).dwt().step(refresh=False)
    O = torch.empty_like(Q)
    ws = torch.zeros(wf.wf_attn_workspace_bytes(Q, k, ng), dtype=torch.uint8, device="cuda")
    wf.wf_sparse_attn(Q, K, V, run.idx, k, Kg, Vg, O, ws)
    at = run.idx.long().view(1, H, k, 1).expand(-1, -1, -1, d)
    Ks, Vs = (torch.cat([t.gather(2, at), e], 2).double() for t, e in ((K, Kg), (V, Vg)))
    R = torch.softmax(Q.double() @ Ks.transpose(2, 3) / d ** 0.5, -1) @ Vs
    one, split = ((x.double() - R).norm().item() for x in (run.O, O))
    assert split <= 1.2 * one
