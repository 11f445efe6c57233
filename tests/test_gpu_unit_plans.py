"""The fused kernel's choice of units a cluster and warpgroups a unit, on both
sides of each line: 64 units with at most 128 KB of candidate rows a unit (one
unit a cluster) and just above (two), one-unit plans with lists of 1022 (one
warpgroup) and 1024 (both).  A step, and the filter and the attention as calls
of their own.

Indices and level sets bit-exact against the planted answer.  Outputs against
the fp64 oracle: the bf16 bound of the other tests; step and separate calls
select the same rows."""
import pytest
import torch

import oracle
from helpers import LibRun, assert_close_out, f64
from paper_2606_00724_gb300 import synth, wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("B,H,d,n,L,k", [
    (2, 32, 128, 2048, 2, 200),  # 512 rows of 256 bytes: one unit a cluster, one warpgroup
    (2, 32, 128, 2056, 2, 201),  # 514: two units, token trim
    (2, 32, 64, 4096, 2, 400),   # 1024 rows of 128 bytes: one unit, both warpgroups
    (2, 32, 64, 4104, 2, 401),   # 1026: two units
    (1, 32, 128, 4088, 2, 400),  # one unit, lists of 1022: one warpgroup
    (1, 32, 128, 4096, 2, 400),  # lists of 1024: both
    (1, 61, 128, 8192, 3, 819),  # an odd number of units in pairs
])
def test_unit_plans(B, H, d, n, L, k):
    w = synth.Workload("unit_plans", B, H, d, n, 32, 32, L, tuple(wf.wf_default_schedule(n, L, k)), "bf16", "iid")
    units = [0, B * H // 2, B * H - 1]
    b = synth.make_batch(w, planted=True, device="cuda", cfg="plans", units=units)
    run = LibRun(b.Q, b.K, b.V, b.Kg, b.Vg, L, w.keep).dwt().step(refresh=False)
    wf.wf_workspace_status(run.ws_step)
    calls = LibRun(b.Q, b.K, b.V, b.Kg, b.Vg, L, w.keep).dwt().filter()
    assert torch.equal(calls.idx, run.idx) and torch.equal(calls.sets, run.sets)
    O = torch.empty_like(b.Q)
    ws = torch.zeros(wf.wf_attn_workspace_bytes(b.Q, k, 32), dtype=torch.uint8, device="cuda")
    wf.wf_sparse_attn(b.Q, b.K, b.V, calls.idx, k, b.Kg, b.Vg, O, ws)
    wf.wf_workspace_status(ws)
    torch.cuda.synchronize()
    for u in units:
        i, h = divmod(u, H)
        got = run.level_sets(u)
        for lev in range(L, -1, -1):
            assert torch.equal(torch.as_tensor(got[lev]).cpu().long(), b.targets[u][lev].cpu().long()), f"{u} {lev}"
        want = oracle.sparse_attn(f64(b.Q[i, h]), f64(b.K[i, h]), f64(b.V[i, h]), run.idx[u].cpu().numpy(),
                                  f64(b.Kg[i, h]), f64(b.Vg[i, h]))
        assert_close_out(f64(run.O[i, h]), want, torch.bfloat16)
        assert_close_out(f64(O[i, h]), want, torch.bfloat16)
