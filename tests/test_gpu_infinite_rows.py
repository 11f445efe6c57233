"""Rows whose logits are -inf for every query (masked keys: infinite, or the
type's lowest value, which overflows): their weight is 0, so they rank below
every other row, equal among themselves (lowest position first), and do not
disturb the ranking of the others.  On every filter route: the fused kernels of
both element types and head dims, the grouped one and the kernels per scale.

Selections against the fp64 oracle, bit for bit; the inputs are random, and the
oracle's smallest relative gap at a Top-K boundary is checked to exceed what
fp32 sums of 64 terms can move (2^-17), so that no near-tie decides.

In the attention such a row adds nothing, also where it fills a whole tile or
slice: outputs within the bounds of the other tests."""

import numpy as np
import pytest
import torch

import oracle
from helpers import LibRun, assert_close_out, f64
from paper_2606_00724_gb300 import wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)

DT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _inputs(dtype, H, group, d, n, q, masked, value, seed):
    """Positive queries (a masked key then has -inf logits, not NaN) and keys with `masked` tokens set to value."""
    g = torch.Generator().manual_seed(seed)
    Q = torch.randn(1, H * group, q, d, generator=g).abs().mul(0.7)
    K = torch.randn(1, H, n, d, generator=g)
    K[:, :, masked] = value if value == -float("inf") else torch.finfo(DT[dtype]).min
    return Q.to(DT[dtype]).cuda(), K.to(DT[dtype]).cuda()


def _oracle(Q, K, n, L, keep, bf16):
    """Level sets of one unit in fp64, with the smallest relative gap at a boundary."""
    with np.errstate(all="ignore"):
        pyr = oracle.haar_pyramid_spec32(K.astype(np.float32), L, bf16)
        cand, sets, gap = np.arange(n >> L), {}, np.inf
        for lev in range(L, -1, -1):
            rows = oracle.level(pyr, n, lev)[cand].astype(np.float64) if lev else K[cand]
            if lev == 0 and keep[0] == cand.size:
                sets[0] = cand
                break
            s = Q @ rows.T / np.sqrt(Q.shape[1])
            p = np.exp(s - s.max(1, keepdims=True))
            W = (p / p.sum(1, keepdims=True)).sum(0)
            order = np.argsort(-W, kind="stable")
            a, b = W[order[keep[lev] - 1]], W[order[keep[lev]]] if keep[lev] < W.size else 0.0
            if a > 0:
                gap = min(gap, (a - b) / a)
            kept = np.sort(order[:keep[lev]])
            sets[lev] = cand[kept]
            if lev:
                cand = np.stack([2 * cand[kept], 2 * cand[kept] + 1], 1).reshape(-1)
    return sets, gap


FEW = slice(37, 43)


@pytest.mark.parametrize("dtype,H,group,d,n,q,L,k,masked,value", [
    ("f32", 2, 1, 64, 4096, 3, 2, 512, FEW, -float("inf")),      # one launch
    ("f32", 2, 1, 128, 4096, 40, 2, 513, FEW, "lowest"),         # the 64-row kernels, token trim
    ("f32", 1, 1, 64, 256, 1, 1, 250, slice(100, 160), -float("inf")),  # more kept than have a weight
    ("f32", 1, 1, 64, 16640, 3, 1, 1001, FEW, -float("inf")),    # the kernels per scale
    ("f32", 1, 3, 128, 1024, 5, 2, 128, slice(64, 192), -float("inf")),  # grouped heads: the same, whole tiles masked
    ("bf16", 2, 1, 128, 1024, 3, 2, 128, FEW, -float("inf")),    # the fused kernel
    ("bf16", 1, 1, 128, 256, 1, 1, 250, slice(100, 160), -float("inf")),
    ("bf16", 2, 1, 64, 1024, 3, 2, 128, FEW, "lowest"),
    ("bf16", 1, 4, 128, 1024, 5, 2, 128, FEW, -float("inf")),    # the grouped kernel
    ("bf16", 1, 4, 64, 256, 1, 1, 250, slice(100, 160), -float("inf")),
    ("bf16", 2, 1, 128, 1024, 32, 2, 250, slice(300, 940), -float("inf")),  # no padded query rows, most rows masked
    ("bf16", 1, 1, 128, 1024, 40, 1, 500, slice(0, 640), -float("inf")),    # blocks of more than 32 rows
    ("bf16", 1, 1, 128, 16640, 3, 1, 1001, FEW, -float("inf")),  # the kernels per scale
    ("bf16", 1, 1, 128, 16640, 40, 1, 4100, slice(0, 10000), -float("inf")),
])
def test_filter_ranks_rows_without_weight_last(dtype, H, group, d, n, q, L, k, masked, value):
    Q, K = _inputs(dtype, H, group, d, n, q, masked, value, seed=k + d + q)
    keep = wf.wf_default_schedule(n, L, k)
    run = LibRun(Q, K, K, None, None, L, keep).dwt().filter()
    torch.cuda.synchronize()
    for u in range(H):
        want, gap = _oracle(f64(Q[0, u * group:(u + 1) * group]).reshape(-1, d), f64(K[0, u]), n, L, keep,
                            dtype == "bf16")
        assert gap > 2.0 ** -17
        got = run.level_sets(u)
        for lev in range(L, -1, -1):
            assert np.array_equal(np.asarray(got[lev]), want[lev]), f"unit {u} scale {lev}"


def _attention(Q, K, V, group):
    """softmax(Q K^T / sqrt d) V in fp64, on the device."""
    Q, K, V = Q.double(), K.double().repeat_interleave(group, 1), V.double().repeat_interleave(group, 1)
    return torch.softmax(Q @ K.transpose(2, 3) / Q.shape[3] ** 0.5, -1) @ V


@pytest.mark.parametrize("dtype,H,group,d,q,n,k,masked", [
    ("bf16", 2, 1, 128, 9, 2048, 512, slice(120, 420)),    # the fused kernel's attention: whole slices masked
    ("bf16", 2, 1, 64, 32, 2048, 512, slice(0, 300)),
    ("bf16", 90, 1, 128, 32, 2048, 512, slice(0, 300)),    # the first tiles of a longer slice
    ("bf16", 2, 1, 128, 32, 16384, 8200, slice(0, 4000)),  # the split kernels: keys on the TMEM lanes
    ("bf16", 2, 4, 128, 32, 2048, 700, slice(0, 300)),     # query rows on the TMEM lanes
    ("bf16", 2, 2, 64, 40, 2048, 512, slice(60, 300)),     # CUDA cores
    ("f32", 2, 1, 128, 9, 2048, 512, slice(60, 300)),
])
def test_attention_ignores_rows_without_weight(dtype, H, group, d, q, n, k, masked):
    Q, K = _inputs(dtype, H, group, d, n, q, masked, -float("inf"), seed=k + d + q)
    V = torch.randn(1, H, n, d, generator=torch.Generator().manual_seed(k)).to(DT[dtype]).cuda()
    idx = torch.arange(k, dtype=torch.int32, device="cuda").repeat(H, 1)
    O = torch.empty_like(Q)
    ws = torch.zeros(wf.wf_attn_workspace_bytes(Q, k, 0), dtype=torch.uint8, device="cuda")
    wf.wf_sparse_attn(Q, K, V, idx, k, None, None, O, ws)
    wf.wf_workspace_status(ws)
    assert_close_out(f64(O), f64(_attention(Q, K[:, :, :k], V[:, :, :k], group)), DT[dtype])


@pytest.mark.parametrize("dtype,d,q", [("f32", 64, 3), ("f32", 128, 40), ("bf16", 128, 3), ("bf16", 64, 32)])
def test_step_that_keeps_rows_without_weight(dtype, d, q):
    n, L, k = 512, 1, 500
    Q, K = _inputs(dtype, 2, 1, d, n, q, slice(100, 300), -float("inf"), seed=d + q)
    V = torch.randn(1, 2, n, d, generator=torch.Generator().manual_seed(q)).to(DT[dtype]).cuda()
    run = LibRun(Q, K, V, None, None, L, wf.wf_default_schedule(n, L, k)).dwt().step(refresh=False)
    wf.wf_workspace_status(run.ws_step)
    at = run.idx.long().view(1, 2, k, 1).expand(-1, -1, -1, d)
    assert_close_out(f64(run.O), f64(_attention(Q, K.gather(2, at), V.gather(2, at), 1)), DT[dtype])
