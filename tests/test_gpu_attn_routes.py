"""wf_sparse_attn on the fused kernel's attention (bf16, one query head a key
head, at most 32 query rows) at its edges: fewer keys than CTAs in the
cluster, ragged slices, clusters of one to eight CTAs, lists of 8192 tokens
(its largest), and on the split kernels (longer lists, more units than
clusters at once); unsorted, repeated and out-of-range tokens (clamped), an
explicit scale, [B, rows, H, d] strides, both head dims.  (Two units a cluster:
test_gpu_two_units.py.)  Outputs against the fp64 oracle: O is rounded to
bf16 once, and the split kernels round P as well (relative 2^-8 each, the
weights' errors averaging below their bound): the bf16 bound of the other
tests.  The fused attention's own error is held to the rounding of O."""
import numpy as np
import pytest
import torch

import oracle
from helpers import assert_close_out, f64
from paper_2606_00724_gb300 import wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("B,H,d,q,n,k,ng,scale,bshd", [
    (1, 1, 128, 1, 64, 1, 0, 0.0, False),
    (1, 2, 64, 32, 256, 3, 2, 0.0, True),
    (2, 3, 128, 17, 2048, 333, 5, 0.25, True),
    (2, 32, 128, 32, 4096, 517, 32, 0.0, False),   # one unit a cluster of two CTAs
    (1, 32, 64, 31, 8192, 1000, 7, 0.2, True),
    (1, 2, 128, 32, 16384, 8192, 3, 0.0, False),   # the largest list
    (1, 1, 128, 32, 16384, 8193, 0, 0.0, False),   # the split kernels: a longer one
    (3, 60, 128, 5, 1024, 200, 0, 0.0, False),     # and more units than clusters fit at once
])
def test_attention_route(B, H, d, q, n, k, ng, scale, bshd):
    g = torch.Generator(device="cpu").manual_seed(k + d)

    def rn(rows):
        t = torch.randn(B, H, rows, d, generator=g).to(torch.bfloat16).cuda()
        return t.transpose(1, 2).contiguous().transpose(1, 2) if bshd else t

    Q, K, V, Kg, Vg = rn(q), rn(n), rn(n), rn(max(ng, 1)), rn(max(ng, 1))
    idx = torch.randint(0, n, (B * H, k), generator=g, dtype=torch.int32)
    if k > 2:
        idx[0, 0], idx[-1, -1] = -5, n + 7
    O = torch.empty_like(Q)
    ws = torch.zeros(wf.wf_attn_workspace_bytes(Q, k, ng), dtype=torch.uint8, device="cuda")
    wf.wf_sparse_attn(Q, K, V, idx.cuda(), k, Kg if ng else None, Vg if ng else None, O, ws, scale)
    wf.wf_workspace_status(ws)
    torch.cuda.synchronize()
    for u in {0, B * H // 2, B * H - 1}:
        i, h = divmod(u, H)
        # an explicit scale is a factor of the queries
        Qs = f64(Q[i, h]) * (scale * d ** 0.5 if scale else 1.0)
        at = idx[u].numpy().clip(0, n - 1)
        want = oracle.sparse_attn(Qs, f64(K[i, h]), f64(V[i, h]), at, f64(Kg[i, h]) if ng else None,
                                  f64(Vg[i, h]) if ng else None)
        assert_close_out(f64(O[i, h]), want, torch.bfloat16)


@pytest.mark.parametrize("d,q,k,ng,amp", [
    (128, 32, 1024, 18, 2.0),   # peaked rows, three tiles a CTA
    (128, 32, 300, 5, 1.0),     # a tile a CTA
    (128, 9, 4000, 0, 3.0),     # both warpgroups
    (64, 32, 1024, 18, 2.0),
])
def test_attention_keeps_more_than_bf16_weights(d, q, k, ng, amp):
    """|O - R| <= 2^-8 |R| + 2^-15 max |V|: O's rounding to bf16 (8 significant
    bits: half a unit is at most 2^-8 of the value); the weights keep 16 bits
    (two terms, 2^-8 of 2^-8), and the fp32 rounding of a logit below 64 and
    its exponential moves one by less than 2^-16.  Weights rounded to bf16
    miss it by 2^-8 of the largest one's share where |R| is small."""
    g = torch.Generator(device="cpu").manual_seed(k)
    B, H, n = 1, 32, 8192

    def rn(rows, a=1.0):
        return (a * torch.randn(B, H, rows, d, generator=g)).to(torch.bfloat16).cuda()

    Q, K, V, Kg, Vg = rn(q, amp), rn(n), rn(n), rn(max(ng, 1)), rn(max(ng, 1))
    idx = torch.stack([torch.randperm(n, generator=g)[:k].sort().values for _ in range(B * H)]).int().cuda()
    O = torch.empty_like(Q)
    ws = torch.zeros(wf.wf_attn_workspace_bytes(Q, k, ng), dtype=torch.uint8, device="cuda")
    wf.wf_sparse_attn(Q, K, V, idx, k, Kg if ng else None, Vg if ng else None, O, ws)
    wf.wf_workspace_status(ws)
    at = idx.long().view(B, H, k, 1).expand(-1, -1, -1, d)
    Ks, Vs = K.gather(2, at).double(), V.gather(2, at).double()
    if ng:
        Ks, Vs = torch.cat([Ks, Kg.double()], 2), torch.cat([Vs, Vg.double()], 2)
    R = torch.softmax(Q.double() @ Ks.transpose(2, 3) / d ** 0.5, -1) @ Vs
    assert ((O.double() - R).abs() <= 2.0 ** -8 * R.abs() + 2.0 ** -15 * Vs.abs().max()).all()


@pytest.mark.parametrize("H,d,q,n,k,ng,bshd", [
    (160, 128, 32, 1024, 300, 5, False),   # more units than clusters at once
    (32, 128, 17, 16384, 8192, 18, True),  # the fused kernel's largest list
    (96, 128, 32, 2048, 1024, 32, False),  # nine tiles a CTA against three of a split
    (40, 128, 1, 4096, 2500, 0, True),     # one query row
    (512, 128, 3, 256, 1, 0, False),       # one key
])
def test_split_attention_keeps_as_much(H, d, q, n, k, ng, bshd):
    """The calls that the split kernels take over from the fused attention, to
    the same bound (their P has the two terms too): unsorted and repeated
    tokens, [B, rows, H, d] strides."""
    g = torch.Generator().manual_seed(k)

    def rn(rows, a=1.0):
        t = (a * torch.randn(1, H, rows, d, generator=g)).to(torch.bfloat16).cuda()
        return t.transpose(1, 2).contiguous().transpose(1, 2) if bshd else t

    Q, K, V, Kg, Vg = rn(q, 2.0), rn(n), rn(n), rn(max(ng, 1)), rn(max(ng, 1))
    idx = torch.randint(0, n, (H, k), generator=g, dtype=torch.int32).cuda()
    O = torch.empty_like(Q)
    ws = torch.zeros(wf.wf_attn_workspace_bytes(Q, k, ng), dtype=torch.uint8, device="cuda")
    wf.wf_sparse_attn(Q, K, V, idx, k, Kg if ng else None, Vg if ng else None, O, ws)
    wf.wf_workspace_status(ws)
    at = idx.long().view(1, H, k, 1).expand(-1, -1, -1, d)
    Ks, Vs = K.gather(2, at).double(), V.gather(2, at).double()
    if ng:
        Ks, Vs = torch.cat([Ks, Kg.double()], 2), torch.cat([Vs, Vg.double()], 2)
    R = torch.softmax(Q.double() @ Ks.transpose(2, 3) / d ** 0.5, -1) @ Vs
    assert ((O.double() - R).abs() <= 2.0 ** -8 * R.abs() + 2.0 ** -15 * Vs.abs().max()).all()
