"""The calls that are timed: one layer's work of a denoising step, through the entry points of
paper_2606_00724_gb300.wf, over the shapes that the library serves.

A case is one layer: B prompts, H key heads, `group` query heads a key head, n cached tokens of head_dim d,
a block of q query rows, ng generation rows, L scales, k kept tokens.  Inputs are the seeded synthetic layers
of synth.make_batch with a planted answer, as the parity tests use them: every Top-K has a margin at its
boundary, so the selected positions are the same whole numbers for any correct arithmetic.
"""
from __future__ import annotations

import math

import torch

from paper_2606_00724_gb300 import synth, wf

DEVICE = "cuda"
EXACT_LIMIT = 1 << 23  # unit-tokens of a case that exact() takes on

# Generators of synth.py with the options of the repository's workloads.
_EXTRA = {
    "needles": lambda n: {"needles": max(1, n // 128)},
    "rope_spans": lambda n: {"spans": 32, "span_len": 16},
    "clusters": lambda n: {"centroids": 64, "seg_min": 256, "seg_max": 2048, "needle_frac": 0.001,
                           "gap_growth": 2.0 ** 0.5},
    "drift": lambda n: {"period": 4096, "needles": max(1, n // 1024), "gap_growth": 2.0 ** 0.5},
    "iid": lambda n: {},
}


def _case(op, B, H, d, n, q, ng, L, k, dtype="bf16", group=1, kind="clusters", schedule="default", layout="bhsd",
          name=None, **more):
    c = dict(op=op, B=B, H=H, d=d, n=n, q=q, ng=ng, L=L, k=k, dtype=dtype, group=group, kind=kind, schedule=schedule,
             layout=layout, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest call: a short prompt, few heads, fp32.  Latency and launches count.
        _case("step", 1, 4, 64, 1024, 32, 32, 2, 128, "f32", kind="needles", name="step_f32_1k"),
        # fp32 at an ordinary prompt length (the path of callers that keep fp32 caches).
        _case("step", 1, 16, 128, 8192, 32, 32, 3, 819, "f32", kind="iid", name="step_f32_8k"),
        # bf16 with 64-wide heads, a ragged prompt length, caches in [B, rows, H, d] order.
        _case("step", 2, 16, 64, 8200, 32, 32, 3, 821, "bf16", kind="iid", layout="bshd", name="step_bf16_d64_8k"),
        # One layer at the three prompt lengths of the benchmark: 8K with an odd k (a token-level scan), 32K, 128K.
        _case("step", 1, 32, 128, 8192, 32, 32, 3, 819, kind="rope_spans", name="step_bf16_8k"),
        _case("step", 2, 32, 128, 32768, 32, 32, 4, 2048, name="step_bf16_32k"),
        _case("step", 1, 32, 128, 131072, 32, 32, 5, 4096, kind="drift", name="step_bf16_128k"),
        # A step that rebuilds the pyramid first, at the largest batch (every eighth step of the 32-layer stack).
        _case("step", 4, 32, 128, 32768, 32, 32, 4, 1638, kind="iid", refresh=True, name="refresh_step_bf16_32k"),
        # A denoising block of 64 rows, the largest that the calls take.
        _case("step", 1, 32, 128, 16384, 64, 64, 4, 1639, kind="iid", name="step_bf16_q64_16k"),
        # Grouped query heads (28 on 4), the large batch of the benchmark.
        _case("step", 8, 4, 128, 32768, 32, 32, 4, 2048, group=7, name="step_gqa_32k"),
        # The literal path with the db2 basis.
        _case("step_wavelet", 2, 32, 128, 32768, 32, 32, 4, 2048, wavelet=1, name="step_db2_32k"),
        # Filter and attention called one after the other, as a program that looks at the selection does: a ragged
        # prompt, a short last block, [B, rows, H, d] caches.
        _case("stages", 1, 32, 128, 20496, 24, 17, 4, 1025, kind="iid", layout="bshd", name="stages_bf16_20k"),
        # 32 new rows a head into the caches at an unaligned place, with the touched blocks of the pyramid.
        _case("update", 2, 32, 128, 32768, 32, 0, 4, 2048, kind="iid", rows=32, pos=12340, name="update_bf16_32k"),
    ]


def draw(rng):
    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    family = rng.choices(["step", "gqa", "wide", "plain", "stages", "wavelet", "update", "build"],
                         [6, 3, 2, 3, 2, 2, 1, 1])[0]
    dtype, d, group = "bf16", 128, 1
    H, B = rng.choice([4, 6, 8, 12, 16, 24, 32]), rng.choice([1, 1, 2, 3, 4])
    # Unit-tokens (B H n) stay at or below those of the family's largest listed case.
    most, lo, hi = 1 << 22, 2048, 131072
    q = 32 if rng.random() < 0.5 else rng.randint(4, 32)
    if family == "gqa":
        H, B, group = rng.choice([2, 4, 8]), rng.choice([1, 2, 4, 8]), rng.choice([2, 3, 4, 7, 8])
        most, hi = 1 << 20, 65536
    elif family == "wide":
        q, most, hi = rng.randint(33, 64), 1 << 19, 32768
    elif family == "plain":  # fp32, or 64-wide heads
        dtype, d = rng.choice([("f32", 64), ("f32", 128), ("bf16", 64)])
        most, lo, hi = 1 << 17, 1024, 16384
    elif family == "stages":
        most, hi = 1 << 19, 32768
    elif family == "wavelet":
        most, hi = 1 << 21, 65536
    while B * H * lo > most:
        B, H = (B - 1, H) if B > 1 else (B, H // 2)
    n = int(log(lo, min(hi, most // (B * H))))
    L = 2 if n < 4096 else 3 if n < 16384 else 4 if n < 65536 else 5
    L = max(2, L + rng.choice([-1, 0, 0, 0]))
    n = max(n >> L, 1) << L
    k = max(64, int(n * log(0.03, 0.12)))
    ng = rng.choice([0, 32, 32, rng.randint(1, 64)])
    kind = rng.choice(["iid", "clusters", "drift"]) if n >= 8192 else "iid"
    layout = rng.choice(["bhsd", "bshd"])
    schedule = "level0" if family in ("step", "gqa") and rng.random() < 0.2 else "default"
    more = {}
    if family == "step" and rng.random() < 0.15:
        more["refresh"] = True
    if family == "wavelet":
        more["wavelet"] = rng.choice([0, 1, 1])
    if family == "update":
        more["rows"] = rng.choice([1, 32, 64, rng.randint(2, 512)])
        more["pos"] = rng.randrange(0, n - more["rows"] + 1)
    op = {"wavelet": "step_wavelet", "stages": "stages", "update": "update", "build": "build"}.get(family, "step")
    return _case(op, B, H, d, n, q, ng, L, k, dtype, group, kind, schedule, layout, **more)


def _keep(case):
    make = wf.wf_level0_schedule if case["schedule"] == "level0" else wf.wf_default_schedule
    return make(case["n"], case["L"], case["k"])


def _layout(case, t):
    """t ([B, H, rows, d]) in the case's memory order."""
    return t.transpose(1, 2).contiguous().transpose(1, 2) if case["layout"] == "bshd" else t


def _inputs(case, seed):
    w = synth.Workload(case["op"], case["B"], case["H"], case["d"], case["n"], case["q"], max(1, case["ng"]),
                       case["L"], tuple(_keep(case)), case["dtype"], case["kind"],
                       extra=_EXTRA[case["kind"]](case["n"]), group=case["group"])
    return synth.make_batch(w, layer=seed, planted=case["op"] not in ("update", "build"), device=DEVICE, cfg="cases")


def prepare(case, seed):
    b = _inputs(case, seed)
    L, op = case["L"], case["op"]
    dt = b.K.dtype
    s = {"op": op, "L": L, "keep": _keep(case), "K": _layout(case, b.K), "V": _layout(case, b.V)}
    B, H, n, d = s["K"].shape
    if op in ("update", "build"):
        s["coeffs"] = torch.zeros(B * H, n - (n >> L), d, dtype=dt, device=DEVICE)
        if op == "update":
            wf.wf_dwt_build(s["K"], L, s["coeffs"])
            g = torch.Generator(device=DEVICE).manual_seed(seed)
            s["pos"] = case["pos"]
            s["Kn"], s["Vn"] = (torch.randn(B, H, case["rows"], d, generator=g, device=DEVICE).to(dt)
                                for _ in range(2))
        return s
    s["Q"] = _layout(case, b.Q)
    s["Kg"], s["Vg"] = (_layout(case, b.Kg), _layout(case, b.Vg)) if case["ng"] else (None, None)
    s["O"] = torch.empty_like(s["Q"])
    s["idx"] = torch.empty(B * H, s["keep"][0], dtype=torch.int32, device=DEVICE)
    if op == "step_wavelet":
        s["wavelet"] = case["wavelet"]
        s["top"] = torch.empty(B, H, n >> L, d, dtype=dt, device=DEVICE)
        wf.wf_wavelet_approx(s["K"], L, s["wavelet"], s["top"])
        size = wf.wf_step_wavelet_workspace_bytes(s["Q"], s["K"], L, s["keep"], s["wavelet"], case["ng"])
    else:
        s["refresh"] = bool(case.get("refresh"))
        s["coeffs"] = torch.zeros(B * H, n - (n >> L), d, dtype=dt, device=DEVICE)
        if not s["refresh"]:
            wf.wf_dwt_build(s["K"], L, s["coeffs"])
        size = wf.wf_step_workspace_bytes(s["Q"], s["K"], L, s["keep"], case["ng"])
        if op == "stages":
            size = wf.wf_filter_workspace_bytes(s["Q"], s["K"], L, s["keep"])
            s["attn_ws"] = torch.zeros(wf.wf_attn_workspace_bytes(s["Q"], s["keep"][0], case["ng"]),
                                       dtype=torch.uint8, device=DEVICE)
    s["ws"] = torch.zeros(size, dtype=torch.uint8, device=DEVICE)
    return s


def run(s):
    op = s["op"]
    if op == "build":
        wf.wf_dwt_build(s["K"], s["L"], s["coeffs"])
        return {"coeffs": s["coeffs"]}
    if op == "update":
        wf.wf_cache_update(s["Kn"], s["Vn"], s["K"], s["V"], s["pos"], s["L"], s["coeffs"])
        return {"K": s["K"], "V": s["V"], "coeffs": s["coeffs"]}
    if op == "stages":
        wf.wf_filter(s["Q"], s["coeffs"], s["K"], s["L"], s["keep"], s["idx"], s["ws"])
        wf.wf_sparse_attn(s["Q"], s["K"], s["V"], s["idx"], s["keep"][0], s["Kg"], s["Vg"], s["O"], s["attn_ws"])
    elif op == "step_wavelet":
        wf.wf_step_wavelet(s["Q"], s["top"], s["K"], s["V"], s["Kg"], s["Vg"], s["L"], s["keep"], s["wavelet"],
                           s["idx"], s["O"], s["ws"])
    else:
        wf.wf_step(s["Q"], s["K"], s["V"], s["Kg"], s["Vg"], s["coeffs"], s["refresh"], s["L"], s["keep"], s["idx"],
                   s["O"], s["ws"])
        if s["refresh"]:
            return {"O": s["O"], "idx": s["idx"], "coeffs": s["coeffs"]}
    return {"O": s["O"], "idx": s["idx"]}


def work(case):
    B, H, d, n, q, ng, L, G = (case[x] for x in ("B", "H", "d", "n", "q", "ng", "L", "group"))
    row = d * (4 if case["dtype"] == "f32" else 2)
    U = B * H
    if case["op"] == "build":
        return {"bytes": U * row * (n + n - (n >> L)), "flops": 2 * U * d * (n - (n >> L))}
    if case["op"] == "update":
        R, pos = case["rows"], case["pos"]
        blocks = ((pos + R - 1) >> L) - (pos >> L) + 1
        # New K and V rows read and written, the blocks' other rows read, their coefficients written.
        rows = 4 * R + ((blocks << L) - R) + blocks * ((1 << L) - 1)
        return {"bytes": U * row * rows, "flops": 2 * U * d * blocks * ((1 << L) - 1)}
    keep = _keep(case)
    k = keep[0]
    cand = {L: n >> L, **{b: 2 * keep[b + 1] for b in range(L)}}
    scored = sum(cand[b] for b in range(1, L + 1)) + (cand[0] if k < cand[0] else 0)
    flops = U * G * q * d * (2 * scored + 4 * (k + ng))
    rows = 2 * G * q + 2 * ng  # Q, O, the generation rows
    if case["op"] == "step_wavelet":
        # The cached top rows, every key that some scale's transform reads (the finer scales' blocks lie inside the
        # first gathered scale's), and the value rows.  The key rows that are attended lie in those blocks too.
        taps = 2 if case["wavelet"] == 0 else 4
        rows += cand[L] + (cand[L - 1] << (L - 1)) + k
        flops += U * d * 2 * taps * sum(cand[b] << b for b in range(1, L))
    elif case.get("refresh"):
        rows += n + (n - (n >> L)) + k  # keys read and the pyramid written once, value rows
        flops += 2 * U * d * (n - (n >> L))
    else:
        # Coefficient rows of the candidates, token candidates (they hold the selected rows) or selected key rows,
        # value rows.
        rows += sum(cand[b] for b in range(1, L + 1)) + (cand[0] if k < cand[0] else k) + k
    return {"bytes": U * (rows * row + 4 * k), "flops": flops}


def tolerance(case):
    if case["op"] in ("build", "update"):
        return "exact"  # the transform's arithmetic is specified to the bit
    return {"rel": 1e-5} if case["dtype"] == "f32" else {"rel": 1e-2}


# ---------------------------------------------------------------------------
# The same in 64 bits.
# ---------------------------------------------------------------------------
_R3 = math.sqrt(3.0)
_TAPS = ([1 / math.sqrt(2)] * 2, [x / (4 * math.sqrt(2)) for x in (1 + _R3, 3 + _R3, 3 - _R3, 1 - _R3)])


def _analyse(x, taps):
    """One level of the periodic transform along the rows of x."""
    return sum(h * x.roll(-i, -2)[..., 0::2, :] for i, h in enumerate(taps))


def _select(Q, rows, kb):
    """Places of the kb largest column sums of softmax(Q rows^T / sqrt d), ascending."""
    W = torch.softmax(Q @ rows.T / math.sqrt(Q.shape[1]), dim=1).sum(0)
    return torch.sort(W, descending=True, stable=True).indices[:kb].sort().values


def _filter(case, keep, Q, K, dt):
    """mu^0 of one unit; the rows that are scored are rounded to the storage type, as the calls define them."""
    L = case["L"]
    taps = _TAPS[case.get("wavelet", 0)]
    literal = case["op"] == "step_wavelet"
    pyramid = [K]
    for _ in range(L):
        pyramid.append(_analyse(pyramid[-1], taps))
    cand = torch.arange(case["n"] >> L, device=K.device)
    for b in range(L, 0, -1):
        if literal and b < L:
            rows = K.view(-1, 1 << b, K.shape[1])[cand].reshape(-1, K.shape[1])
            for _ in range(b):
                rows = _analyse(rows, taps)
        else:
            rows = pyramid[b][cand]
        kept = cand[_select(Q, rows.to(dt).double(), keep[b])]
        cand = torch.stack([2 * kept, 2 * kept + 1], 1).reshape(-1)
    return cand[_select(Q, K[cand], keep[0])] if keep[0] < cand.numel() else cand


def exact(case, seed):
    if case["B"] * case["H"] * case["n"] > EXACT_LIMIT:
        return None
    b = _inputs(case, seed)
    B, H, n, d = b.K.shape
    L, G, dt = case["L"], case["group"], b.K.dtype
    K = b.K.double()
    out = {}
    if case["op"] == "update":
        g = torch.Generator(device=DEVICE).manual_seed(seed)
        Kn, Vn = (torch.randn(B, H, case["rows"], d, generator=g, device=DEVICE).to(dt) for _ in range(2))
        at = slice(case["pos"], case["pos"] + case["rows"])
        V = b.V
        V[:, :, at] = Vn
        K[:, :, at] = Kn.double()
        out = {"K": K, "V": V}
    if case["op"] in ("update", "build") or case.get("refresh"):
        levels = [K]
        for _ in range(L):
            levels.append(_analyse(levels[-1], _TAPS[0]))
        out["coeffs"] = torch.cat(levels[1:], dim=2).reshape(B * H, n - (n >> L), d)
        if case["op"] in ("update", "build"):
            return out
    keep = _keep(case)
    out["O"] = torch.empty(b.Q.shape, dtype=torch.float64, device=DEVICE)
    out["idx"] = torch.empty(B * H, keep[0], dtype=torch.int32, device=DEVICE)
    for i in range(B):
        for h in range(H):
            Q = b.Q[i, h * G:(h + 1) * G].double().reshape(-1, d)
            mu = _filter(case, keep, Q, K[i, h], dt)
            Ks, Vs = K[i, h, mu], b.V[i, h, mu].double()
            if case["ng"]:
                Ks, Vs = torch.cat([Ks, b.Kg[i, h].double()]), torch.cat([Vs, b.Vg[i, h].double()])
            out["O"][i, h * G:(h + 1) * G] = (torch.softmax(Q @ Ks.T / math.sqrt(d), 1) @ Vs).view(G, -1, d)
            out["idx"][i * H + h] = mu
    return out
