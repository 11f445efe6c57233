"""The failure path of the tensor-core kernels' bounded waits, driven through
the test-only control of include/wf_testing.h: the first wait of every CTA
waits on a barrier that nothing completes, with a short bound, so it gives
up.  The call must report WF_ERR_TIMEOUT through the workspace status word,
write nothing outside its outputs, and leave the context usable: the next
normal call matches the oracle.  Small layers only (mostly two or four units)."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from helpers import assert_close_out, f64
from paper_2606_00724_gb300 import synth, wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

WF_ERR_TIMEOUT = -7
GUARD = 64          # guard rows / words on each side of an output
SENTINEL = -12288.0  # exact in bf16


def _small_layer(n=4096, levels=3, k=512):
    w = dataclasses.replace(synth.WORKLOADS["c3"], name=f"wait_failure_n{n}", batch=1, heads=4, n=n, levels=levels,
                            keep=tuple(int(x) for x in oracle.default_schedule(n, levels, k)))
    b = synth.make_batch(w, planted=True, device="cpu", cfg="c3")
    return w, dataclasses.replace(b, Q=b.Q.cuda(), K=b.K.cuda(), V=b.V.cuda(), Kg=b.Kg.cuda(), Vg=b.Vg.cuda())


def _guarded_out(Q):
    """O as a view into a buffer with GUARD sentinel rows before and after
    each head's rows."""
    B, H, q, d = Q.shape
    full = torch.full((B, H, q + 2 * GUARD, d), SENTINEL, dtype=Q.dtype, device=Q.device)
    return full, full[:, :, GUARD:GUARD + q, :]


def _guarded_idx(units, k, device):
    full = torch.full((units * k + 2 * GUARD,), -7, dtype=torch.int32, device=device)
    return full, full[GUARD:GUARD + units * k].view(units, k)


def _guards_intact(O_full, idx_full):
    g = O_full[:, :, :GUARD].float(), O_full[:, :, -GUARD:].float()
    assert torch.all(g[0] == SENTINEL) and torch.all(g[1] == SENTINEL), "write outside O"
    assert torch.all(idx_full[:GUARD] == -7) and torch.all(idx_full[-GUARD:] == -7), "write outside idx"


def _oracle_unit(w, batch, u):
    b, h = divmod(u, w.heads)
    Q, K, V, Kg, Vg = (f64(t[b, h]) for t in (batch.Q, batch.K, batch.V, batch.Kg, batch.Vg))
    pyr = oracle.haar_pyramid_spec32(K.astype(np.float32), w.levels, True)
    mu0 = oracle.filter(Q, pyr, K, w.n, w.levels, np.array(w.keep))
    return mu0, oracle.sparse_attn(Q, K, V, mu0, Kg, Vg)


# One unit per cluster, with lists of 512 (4K tokens: one compute warpgroup)
# and of 2048 (32K: both).
@pytest.mark.parametrize("n,levels,k,check", [(4096, 3, 512, 4), (32768, 4, 2048, 2)])
def test_fused_step_wait_gives_up_then_recovers(n, levels, k, check):
    w, batch = _small_layer(n, levels, k)
    keep = list(w.keep)
    coeffs = torch.empty(wf.wf_coeffs_bytes(batch.K, w.levels), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(wf.wf_step_workspace_bytes(batch.Q, batch.K, w.levels, keep, w.ng), dtype=torch.uint8,
                     device="cuda")
    O_full, O = _guarded_out(batch.Q)
    idx_full, idx = _guarded_idx(w.units, w.k, "cuda")
    wf.wf_dwt_build(batch.K, w.levels, coeffs)
    try:
        wf.wf_testing_set_wait_failure(True, 100_000)  # ~50 us at 2 GHz
        wf.wf_step(batch.Q, batch.K, batch.V, batch.Kg, batch.Vg, coeffs, False, w.levels, keep, idx, O, ws)
        with pytest.raises(wf.WfError) as ei:
            wf.wf_workspace_status(ws)
        assert ei.value.status == WF_ERR_TIMEOUT
    finally:
        wf.wf_testing_set_wait_failure(False, 0)
    torch.cuda.synchronize()
    _guards_intact(O_full, idx_full)
    # The status word was cleared by the report; a normal call is exact.
    wf.wf_step(batch.Q, batch.K, batch.V, batch.Kg, batch.Vg, coeffs, False, w.levels, keep, idx, O, ws)
    wf.wf_workspace_status(ws)
    torch.cuda.synchronize()
    _guards_intact(O_full, idx_full)
    for u in range(check):
        mu0, O_ref = _oracle_unit(w, batch, u)
        assert np.array_equal(idx[u].cpu().numpy(), mu0), f"unit {u}"
        assert_close_out(f64(O[0, u]), O_ref, torch.bfloat16)


def test_tensor_core_attention_wait_gives_up_then_recovers():
    w, batch = _small_layer()
    g = torch.Generator(device="cpu").manual_seed(5)
    idx_list = torch.stack([torch.randperm(w.n, generator=g)[: w.k].sort().values for _ in range(w.units)])
    idx_list = idx_list.to(torch.int32).cuda()
    ws = torch.zeros(wf.wf_attn_workspace_bytes(batch.Q, w.k, w.ng), dtype=torch.uint8, device="cuda")
    O_full, O = _guarded_out(batch.Q)
    try:
        wf.wf_testing_set_wait_failure(True, 100_000)
        wf.wf_sparse_attn(batch.Q, batch.K, batch.V, idx_list, w.k, batch.Kg, batch.Vg, O, ws)
        with pytest.raises(wf.WfError) as ei:
            wf.wf_workspace_status(ws)
        assert ei.value.status == WF_ERR_TIMEOUT
    finally:
        wf.wf_testing_set_wait_failure(False, 0)
    torch.cuda.synchronize()
    g0, g1 = O_full[:, :, :GUARD].float(), O_full[:, :, -GUARD:].float()
    assert torch.all(g0 == SENTINEL) and torch.all(g1 == SENTINEL), "write outside O"
    wf.wf_sparse_attn(batch.Q, batch.K, batch.V, idx_list, w.k, batch.Kg, batch.Vg, O, ws)
    wf.wf_workspace_status(ws)
    torch.cuda.synchronize()
    for u in range(w.units):
        b, h = divmod(u, w.heads)
        Q, K, V, Kg, Vg = (f64(t[b, h]) for t in (batch.Q, batch.K, batch.V, batch.Kg, batch.Vg))
        ref = oracle.sparse_attn(Q, K, V, idx_list[u].cpu().numpy(), Kg, Vg)
        assert_close_out(f64(O[b, h]), ref, torch.bfloat16)



def test_grouped_filter_wait_gives_up_then_recovers():
    # wf_step on grouped query heads (the grouped filter kernel, then the
    # tensor-core attention) under the same stalled first wait: the status
    # word reports WF_ERR_TIMEOUT, nothing is written outside idx and O, and
    # the next normal call matches the oracle.
    n, levels, k = 4096, 3, 512
    w = dataclasses.replace(synth.WORKLOADS["g1"], name="wait_failure_gqa", batch=1, heads=2, n=n, levels=levels,
                            keep=tuple(int(x) for x in oracle.default_schedule(n, levels, k)))
    b = synth.make_batch(w, planted=True, device="cpu", cfg="g1")
    batch = dataclasses.replace(b, Q=b.Q.cuda(), K=b.K.cuda(), V=b.V.cuda(), Kg=b.Kg.cuda(), Vg=b.Vg.cuda())
    keep = list(w.keep)
    G = w.group
    coeffs = torch.empty(wf.wf_coeffs_bytes(batch.K, w.levels), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(wf.wf_step_workspace_bytes(batch.Q, batch.K, w.levels, keep, w.ng), dtype=torch.uint8,
                     device="cuda")
    O_full, O = _guarded_out(batch.Q)
    idx_full, idx = _guarded_idx(w.units, w.k, "cuda")
    wf.wf_dwt_build(batch.K, w.levels, coeffs)
    try:
        wf.wf_testing_set_wait_failure(True, 100_000)
        wf.wf_step(batch.Q, batch.K, batch.V, batch.Kg, batch.Vg, coeffs, False, w.levels, keep, idx, O, ws)
        with pytest.raises(wf.WfError) as ei:
            wf.wf_workspace_status(ws)
        assert ei.value.status == WF_ERR_TIMEOUT
    finally:
        wf.wf_testing_set_wait_failure(False, 0)
    torch.cuda.synchronize()
    _guards_intact(O_full, idx_full)
    wf.wf_step(batch.Q, batch.K, batch.V, batch.Kg, batch.Vg, coeffs, False, w.levels, keep, idx, O, ws)
    wf.wf_workspace_status(ws)
    torch.cuda.synchronize()
    _guards_intact(O_full, idx_full)
    for u in range(w.units):
        bb, h = divmod(u, w.heads)
        Qh = f64(batch.Q[bb, h * G:(h + 1) * G])
        K, V, Kg, Vg = (f64(t[bb, h]) for t in (batch.K, batch.V, batch.Kg, batch.Vg))
        pyr = oracle.haar_pyramid_spec32(K.astype(np.float32), w.levels, True)
        mu0 = oracle.filter_gqa(Qh, pyr, K, w.n, w.levels, np.array(w.keep))
        assert np.array_equal(idx[u].cpu().numpy(), mu0), f"unit {u}"
        assert_close_out(f64(O[bb, h * G:(h + 1) * G]), oracle.sparse_attn_gqa(Qh, K, V, mu0, Kg, Vg), torch.bfloat16)


def test_two_unit_step_wait_gives_up_then_recovers():
    # 64 units with more than 128 KB of candidate rows each: two units a cluster.
    n, levels, k = 8192, 3, 819
    w = dataclasses.replace(synth.WORKLOADS["c3"], name="wait_failure_two", batch=2, heads=32, n=n, levels=levels,
                            keep=tuple(int(x) for x in oracle.default_schedule(n, levels, k)))
    b = synth.make_batch(w, planted=True, device="cuda", cfg="c3", units=[0, 63])
    keep = list(w.keep)
    coeffs = torch.empty(wf.wf_coeffs_bytes(b.K, levels), dtype=torch.uint8, device="cuda")
    ws = torch.zeros(wf.wf_step_workspace_bytes(b.Q, b.K, levels, keep, w.ng), dtype=torch.uint8, device="cuda")
    O_full, O = _guarded_out(b.Q)
    idx_full, idx = _guarded_idx(w.units, w.k, "cuda")
    wf.wf_dwt_build(b.K, levels, coeffs)
    call = lambda: wf.wf_step(b.Q, b.K, b.V, b.Kg, b.Vg, coeffs, False, levels, keep, idx, O, ws)
    try:
        wf.wf_testing_set_wait_failure(True, 100_000)
        call()
        with pytest.raises(wf.WfError) as ei:
            wf.wf_workspace_status(ws)
        assert ei.value.status == WF_ERR_TIMEOUT
    finally:
        wf.wf_testing_set_wait_failure(False, 0)
    torch.cuda.synchronize()
    _guards_intact(O_full, idx_full)
    call()
    wf.wf_workspace_status(ws)
    torch.cuda.synchronize()
    _guards_intact(O_full, idx_full)
    for u in (0, 63):
        mu0, O_ref = _oracle_unit(w, b, u)
        assert np.array_equal(idx[u].cpu().numpy(), mu0), f"unit {u}"
        assert_close_out(f64(O[u // 32, u % 32]), O_ref, torch.bfloat16)


@pytest.mark.parametrize("H,group,q,n,k", [
    (2, 2, 16, 4096, 512),      # grouped heads, 32 stacked rows: keys on the TMEM lanes
    (2, 1, 32, 16384, 8200),    # a list beyond the fused attention's
    (16, 1, 32, 16384, 8192),   # and one that takes the split kernel as the faster route: P in two terms
])
def test_split_attention_wait_gives_up_then_recovers(H, group, q, n, k):
    d = 128
    g = torch.Generator().manual_seed(k)
    rn = lambda heads, rows: torch.randn(1, heads, rows, d, generator=g).to(torch.bfloat16).cuda()
    Q, K, V = rn(H * group, q), rn(H, n), rn(H, n)
    idx = torch.stack([torch.randperm(n, generator=g)[:k] for _ in range(H)]).int().cuda()
    ws = torch.zeros(wf.wf_attn_workspace_bytes(Q, k, 0), dtype=torch.uint8, device="cuda")
    O_full, O = _guarded_out(Q)
    try:
        wf.wf_testing_set_wait_failure(True, 100_000)
        wf.wf_sparse_attn(Q, K, V, idx, k, None, None, O, ws)
        with pytest.raises(wf.WfError) as ei:
            wf.wf_workspace_status(ws)
        assert ei.value.status == WF_ERR_TIMEOUT
    finally:
        wf.wf_testing_set_wait_failure(False, 0)
    torch.cuda.synchronize()
    edges = O_full[:, :, :GUARD].float(), O_full[:, :, -GUARD:].float()
    assert torch.all(edges[0] == SENTINEL) and torch.all(edges[1] == SENTINEL), "write outside O"
    wf.wf_sparse_attn(Q, K, V, idx, k, None, None, O, ws)
    wf.wf_workspace_status(ws)
    at = idx.long().view(1, H, k, 1).expand(-1, -1, -1, d)
    Ks, Vs = (t.gather(2, at).double().repeat_interleave(group, 1) for t in (K, V))
    R = torch.softmax(Q.double() @ Ks.transpose(2, 3) / d ** 0.5, -1) @ Vs
    assert_close_out(f64(O), f64(R), torch.bfloat16)
