"""The instances with two units a cluster (one compute warpgroup a unit) of the
calls that prefer one: the filter and the attention as calls of their own and
the literal path take two units a cluster only at unit counts between half and
two thirds of the SMs (80 units on 152 SMs: clusters of three CTAs for two
units against one CTA a unit).  Even and odd counts (the last cluster then has
one unit), both head dims, handed-in token lists, a stabiliser that is raised
in a later tile, token trim.

Indices and level sets bit-exact against the planted answer and the oracle;
outputs within the bf16 bound of the other tests."""
import numpy as np
import pytest
import torch

import oracle
from helpers import LibRun, assert_close_out, f64
from paper_2606_00724_gb300 import synth, wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)


def _units(H):
    return [0, 1, H // 2, H - 1]


@pytest.mark.parametrize("H,d,q,n,L,k", [
    (80, 128, 32, 2048, 2, 205),   # token trim
    (81, 128, 17, 2048, 2, 256),
    (80, 64, 32, 4096, 3, 410),
    (81, 64, 5, 2048, 1, 301),
])
def test_filter(H, d, q, n, L, k):
    w = synth.Workload("two_units", 1, H, d, n, q, 1, L, tuple(wf.wf_default_schedule(n, L, k)), "bf16", "iid")
    b = synth.make_batch(w, planted=True, device="cuda", cfg="two", units=_units(H))
    run = LibRun(b.Q, b.K, b.V, None, None, L, w.keep).dwt().filter()
    torch.cuda.synchronize()
    for u in _units(H):
        got = run.level_sets(u)
        for lev in range(L, -1, -1):
            assert np.array_equal(got[lev], b.targets[u][lev].cpu().numpy()), f"unit {u} scale {lev}"


@pytest.mark.parametrize("H,d,q,n,k,ng,jump", [
    (80, 128, 32, 4096, 500, 18, 1.0),   # two tiles a unit and CTA
    (81, 128, 32, 4096, 1000, 5, 6.0),   # three, raised in the later ones
    (80, 64, 32, 4096, 1000, 0, 6.0),
    (81, 64, 9, 4096, 300, 32, 1.0),
])
def test_attention(H, d, q, n, k, ng, jump):
    """jump: the factor of the logits from the second tile of 128 keys of a
    slice on, so that they exceed the first tile's by more than 2^64."""
    g = torch.Generator().manual_seed(k)
    rn = lambda rows, a=1.0: (a * torch.randn(1, H, rows, d, generator=g)).to(torch.bfloat16).cuda()
    Q, K, V, Kg, Vg = rn(q, 3.0), rn(n, 3.0), rn(n), rn(max(ng, 1)), rn(max(ng, 1))
    idx = torch.stack([torch.randperm(n, generator=g)[:k] for _ in range(H)]).int().cuda()
    if jump != 1.0:
        slice_rows = -(-(k + ng) // 3)
        late = (torch.arange(k) % slice_rows) >= 128
        at = idx[:, late.cuda()].long().view(1, H, -1, 1).expand(-1, -1, -1, d)
        K.scatter_(2, at, (K.gather(2, at).float() * jump).to(torch.bfloat16))
    O = torch.empty_like(Q)
    ws = torch.zeros(wf.wf_attn_workspace_bytes(Q, k, ng), dtype=torch.uint8, device="cuda")
    wf.wf_sparse_attn(Q, K, V, idx, k, Kg if ng else None, Vg if ng else None, O, ws)
    wf.wf_workspace_status(ws)
    at = idx.long().view(1, H, k, 1).expand(-1, -1, -1, d)
    Ks, Vs = K.gather(2, at).double(), V.gather(2, at).double()
    if ng:
        Ks, Vs = torch.cat([Ks, Kg.double()], 2), torch.cat([Vs, Vg.double()], 2)
    s = Q.double() @ Ks.transpose(2, 3) / d ** 0.5
    if jump != 1.0:  # the case is what it says: some row's later tile is above its first by more than 64 in log2
        first, rest = s[..., :128].amax(-1), s[..., 128:-(-(k + ng) // 3)].amax(-1)
        assert ((rest - first) * 1.4427 > 64).any()
    assert_close_out(f64(O), f64(torch.softmax(s, -1) @ Vs), torch.bfloat16)


@pytest.mark.parametrize("H,d,q,n,L,k", [(80, 128, 32, 2048, 2, 205), (81, 64, 9, 2048, 3, 256)])
def test_literal_step(H, d, q, n, L, k):
    w = synth.Workload("two_units_lit", 1, H, d, n, q, 7, L, tuple(wf.wf_default_schedule(n, L, k)), "bf16", "iid")
    b = synth.make_batch(w, planted=True, device="cuda", cfg="two_lit", units=_units(H))
    wv = wf.WF_WAVELET_HAAR
    top = torch.empty(1, H, n >> L, d, dtype=torch.bfloat16, device="cuda")
    wf.wf_wavelet_approx(b.K, L, wv, top)
    ws = torch.zeros(wf.wf_step_wavelet_workspace_bytes(b.Q, b.K, L, w.keep, wv, 7), dtype=torch.uint8, device="cuda")
    idx = torch.empty(H, k, dtype=torch.int32, device="cuda")
    sets = torch.empty(H, sum(w.keep), dtype=torch.int32, device="cuda")
    O = torch.empty_like(b.Q)
    wf.wf_step_wavelet(b.Q, top, b.K, b.V, b.Kg, b.Vg, L, w.keep, wv, idx, O, ws, level_sets=sets)
    wf.wf_workspace_status(ws)
    torch.cuda.synchronize()
    for u in _units(H):
        Qu, Ku = f64(b.Q[0, u]), f64(b.K[0, u])
        mu0, osets = oracle.filter_wavelet(Qu, Ku, L, np.array(w.keep), oracle.HAAR, spec32=True, store_bf16=True,
                                           want_sets=True)
        got = oracle.split_level_sets(sets[u].cpu().numpy(), L, w.keep)
        for lev in range(L, -1, -1):
            assert np.array_equal(got[lev], osets[lev]), f"unit {u} scale {lev}"
        assert np.array_equal(idx[u].cpu().numpy(), mu0)
        want = oracle.sparse_attn(Qu, Ku, f64(b.V[0, u]), mu0, f64(b.Kg[0, u]), f64(b.Vg[0, u]))
        assert_close_out(f64(O[0, u]), want, torch.bfloat16)
