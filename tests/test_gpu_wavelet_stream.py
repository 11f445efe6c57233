"""The streamed approximation kernel (scales 1 to 5) at its edges: lists of one
block (the filter wraps onto it again), runs that end inside a list, long
runs, several blocks a load group and several groups a block, both head
dims, [B, rows, H, d] strides, block indices outside the prompt (every token
clamped to its first or last).  Bit-exact against the fp32 storage rule."""
import numpy as np
import pytest
import torch

import oracle
from paper_2606_00724_gb300 import wf

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("needs a GPU", allow_module_level=True)


@pytest.mark.parametrize("basis", ["haar", "db2"])
@pytest.mark.parametrize("dtype,d,level,m,heads,bshd", [
    (torch.bfloat16, 128, 1, 1, 1, False),
    (torch.bfloat16, 64, 2, 3, 5, True),
    (torch.float32, 128, 3, 2, 2, False),
    (torch.bfloat16, 128, 4, 5, 3, True),
    (torch.bfloat16, 128, 5, 33, 2, False),
    (torch.float32, 64, 5, 9, 1, True),
    (torch.bfloat16, 128, 1, 1501, 70, False),
    (torch.bfloat16, 128, 3, 500, 200, True),
    (torch.bfloat16, 128, 2, 401, 650, False),  # more units than resident CTAs
    (torch.bfloat16, 128, 5, 48, 38, True),     # half of 152 SMs: one output a thread
    (torch.bfloat16, 128, 5, 49, 38, False),    # and just more, runs of 4
    (torch.bfloat16, 64, 5, 23, 200, False),
    (torch.float32, 128, 4, 3, 60, True),
    (torch.bfloat16, 64, 1, 70, 4, False),      # two blocks a load group, a run of one
])
def test_stream_edges(basis, dtype, d, level, m, heads, bshd):
    wv, ov = (wf.WF_WAVELET_HAAR, oracle.HAAR) if basis == "haar" else (wf.WF_WAVELET_DB2, oracle.DB2)
    n = max(m, 4) << level
    g = torch.Generator(device="cuda").manual_seed(m + level)
    K = torch.randn(1, heads, n, d, generator=g, device="cuda").to(dtype)
    if bshd:
        K = K.transpose(1, 2).contiguous().transpose(1, 2)
    r = np.random.default_rng(m)
    cand = r.integers(0, n >> level, (heads, m)).astype(np.int32)
    if m > 2:
        cand[0, 1], cand[-1, -1] = -3, (n >> level) + 2
    out = torch.empty(1, heads, m, d, dtype=dtype, device="cuda")
    wf.wf_wavelet_approx(K, level, wv, out, cand=torch.from_numpy(cand).cuda())
    torch.cuda.synchronize()
    for u in {0, heads // 2, heads - 1}:
        toks = ((cand[u].astype(np.int64) << level)[:, None] + np.arange(1 << level)).reshape(-1).clip(0, n - 1)
        want = oracle.wavelet_approx_spec32(K[0, u].float().cpu().numpy()[toks], ov, level, dtype == torch.bfloat16)
        assert np.array_equal(out[0, u].float().cpu().numpy(), want), f"unit {u}"
