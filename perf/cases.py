"""The attention calls whose speed this repository keeps track of.

One case is one call of one attention layer at one sampling step, made through the classes of `layer.py` the way a
sampler drives them: a dense step, a sparse step (ARM, tile schedule, reordering, pattern-masked attention), a sparse
step with dynamic bandwidth, or a sparse step on host buffers.  Inputs are random with planted structure, a third of
the heads each for the three patterns (as in `synth.py`), drawn on the GPU from the seed.

`listed()` holds the shapes of `synth.WORKLOADS` and a ragged one; `draw(rng)` draws from the ranges they span.
"""
from __future__ import annotations

import math

import torch

from paper_2505_21036_b200 import api, layer

STEPS = 50            # sampling steps; the first tenth are dense, so step 0 is a dense call and step 25 a sparse one
BANDWIDTHS = (0.125, 0.25, 0.5)   # candidates of the dynamic-bandwidth variant
MOST_PAIRS = 1.7e11   # query-key pairs (times D / 128) of the largest listed case
MOST_EXACT = 3e13     # B * H * N^2 * D up to which the 64-bit result takes less than about 20 seconds
SPATIAL, TEMPORAL, TEXTURAL = api.RF_SPATIAL, api.RF_TEMPORAL, api.RF_TEXTURAL


def _case(name, kind, B, H, D, T, fh, fw, L, omega, mode=0, amp=1.5, lse=False, permute=1, key_frame=False, window_2d=False,
          groups=1):
    c = dict(kind=kind, B=B, H=H, D=D, T=T, fh=fh, fw=fw, L=L, omega=omega, mode=mode, amp=amp, lse=lse, permute=permute,
             key_frame=key_frame, window_2d=window_2d, groups=groups)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # a unit-test-sized layer: host time and launch latency are all there is
        _case("tiny_d64", "sparse", 1, 3, 64, 4, 8, 8, 16, 4, mode=1),
        # a short, low-resolution clip with sizes that divide nothing, two prompts in one batch, log-sum-exp wanted
        _case("ragged_d96", "sparse", 2, 5, 96, 7, 19, 27, 77, 7, lse=True),
        # the shortest point of the shape sweep: a few waves of work, sparse and dense
        _case("8x1024_d128", "sparse", 1, 24, 128, 8, 32, 32, 256, 8),
        _case("8x1024_d128_dense", "dense", 1, 24, 128, 8, 32, 32, 256, 8),
        # the same layer for a caller whose tensors live in pinned host memory
        _case("8x1024_d128_host", "host", 1, 24, 128, 8, 32, 32, 256, 8, groups=4),
        # the middle of the sweep with every head choosing its own bandwidth
        _case("16x2040_d128_plus", "plus", 1, 24, 128, 16, 34, 60, 256, 17),
        # the middle of the sweep with the other readings of the patterns: key frame, 2-D window, original token order
        _case("16x2040_d128_options", "sparse", 1, 24, 128, 16, 34, 60, 256, 17, mode=1, permute=0, key_frame=True, window_2d=True),
        # the CogVideoX-shaped layer: weak structure (every head Textural), strong structure (all three patterns), dense
        _case("cogvideox_d64_weak", "sparse", 1, 48, 64, 13, 30, 45, 226, 15, amp=0.5),
        _case("cogvideox_d64", "sparse", 1, 48, 64, 13, 30, 45, 226, 15, amp=2.0, lse=True),
        _case("cogvideox_d64_dense", "dense", 1, 48, 64, 13, 30, 45, 226, 15, amp=2.0),
        # the OpenSoraPlan-shaped layer
        _case("opensoraplan_d96", "sparse", 1, 24, 96, 24, 45, 80, 300, 100, mode=1),
        # the HunyuanVideo-720p-shaped layer, the largest
        _case("hunyuan720p_d128", "sparse", 1, 24, 128, 33, 45, 80, 256, 36),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    while True:
        kind = rng.choice(("sparse", "sparse", "sparse", "dense", "plus", "host"))
        D, T, fh, fw = rng.choice((64, 96, 128)), _log_int(rng, 4, 33), _log_int(rng, 8, 45), _log_int(rng, 8, 80)
        B, H, L = rng.choice((1, 1, 2)), rng.choice((3, 5, 8, 12, 16, 24, 30, 48)), rng.choice((0, 16, 77, 226, 256, 300))
        groups = rng.choice([g for g in (1, 2, 4) if (B * H) % g == 0]) if kind == "host" else 1
        options = kind == "sparse" and rng.random() < 0.25
        c = _case(None, kind, B, H, D, T, fh, fw, L, max(1, int(T * rng.uniform(1.0, 3.0))), mode=rng.choice((0, 1)),
                  amp=2.0 if D == 64 else 1.5, lse=kind in ("sparse", "dense") and rng.random() < 0.3,
                  permute=0 if rng.random() < 0.15 else 1, key_frame=options, window_2d=options, groups=groups)
        # the sample keeps some tokens, a host call stays below what its copies make tedious
        if (T * fh * fw) // c["omega"] >= 48 and _pairs(c) * D / 128 <= MOST_PAIRS * (0.1 if kind == "host" else 0.9):
            return c


def _windows(c):
    return c["T"] // 4, (c["fh"] * c["fw"]) // 4


def _params(c):
    wf, ws = _windows(c)
    return api.make_params(wf, ws, textural_stride=2, sample_mode=c["mode"], sample_stride=c["omega"], alpha=0.9,
                           temporal_permute=c["permute"], spatial_key_first_frame=int(c["key_frame"]),
                           temporal_window_2d=(c["fh"] // 4, c["fw"] // 4) if c["window_2d"] else None)


def _kinds(c):
    third = c["H"] // 3
    return ["frame"] * third + ["position"] * third + ["lowrank"] * (c["H"] - 2 * third)


def _inputs(c, seed):
    """Q, K, V as bf16 [B, H, N, D] on the GPU: N(0, 1), plus each head's planted component on the video tokens of Q and K."""
    B, H, D, T, S = c["B"], c["H"], c["D"], c["T"], c["fh"] * c["fw"]
    N = T * S + c["L"]
    gen = torch.Generator("cuda").manual_seed(seed)
    q, k, v = (torch.empty((B, H, N, D), dtype=torch.bfloat16, device="cuda") for _ in range(3))

    def normal(*shape):
        return torch.randn(shape, generator=gen, device="cuda")

    for b in range(B):
        for h, kind in enumerate(_kinds(c)):
            if kind == "frame":
                pq = pk = normal(T, 1, D) * c["amp"]
            elif kind == "position":
                pq = pk = normal(1, S, D) * c["amp"]
            else:
                w = normal(4, D) * (c["amp"] / 2)
                pq, pk = normal(T, S, 4) @ w, normal(T, S, 4) @ w
            for dst, planted in ((q, pq), (k, pk), (v, None)):
                x = normal(N, D)
                if planted is not None:
                    x[:T * S].view(T, S, D).add_(planted)
                dst[b, h] = x
    return q, k, v


def prepare(case, seed):
    c = case
    shape, params = api.make_shape(c["B"], c["H"], c["D"], c["T"], c["fh"], c["fw"], c["L"]), _params(c)
    q, k, v = _inputs(c, seed)
    if c["kind"] == "host":
        qh, kh, vh = (torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (q, k, v))
        o = torch.empty(q.shape, dtype=q.dtype, pin_memory=True)
        del q, k, v
        return {"attn": layer.HostStagedAttention(shape, params, "cuda", groups=c["groups"]), "qkv": (qh, kh, vh), "o": o, "case": c}
    attn = layer.RainFusionAttention(shape, params, "cuda", bandwidths=BANDWIDTHS if c["kind"] == "plus" else None)
    lse = torch.empty(q.shape[:3], dtype=torch.float32, device="cuda") if c["lse"] else None
    return {"attn": attn, "qkv": (q, k, v), "o": torch.empty_like(q), "lse": lse, "case": c}


def run(state):
    attn, (q, k, v), o, kind = state["attn"], state["qkv"], state["o"], state["case"]["kind"]
    if kind == "host":
        attn(q, k, v, o)
        return {"o": o}
    attn(q, k, v, o, lse=state["lse"], step=0 if kind == "dense" else STEPS // 2, num_steps=STEPS)
    out = {"o": o, "lse": state["lse"]}
    if kind != "dense":
        out["head_class"] = attn.head_class
    if kind == "plus":
        out["head_window"] = attn.head_window
    return out


def _band(n, w):
    """Pairs of an n x n matrix with |i - j| <= w."""
    w = min(w, n - 1)
    return n * (2 * w + 1) - w * (w + 1)


def _pairs(c):
    """Query-key pairs of one call: what the planted patterns keep (all of them for a dense call)."""
    T, S, L = c["T"], c["fh"] * c["fw"], c["L"]
    Nv, N = T * S, T * S + L
    if c["kind"] == "dense":
        return c["B"] * c["H"] * N * N
    wf, ws = _windows(c)
    if c["kind"] == "plus":
        wf, ws = int(BANDWIDTHS[0] * T), int(BANDWIDTHS[0] * S)
    text = Nv * L + L * N
    spatial = _band(T, wf)
    if c["key_frame"]:
        spatial += max(T - wf - 1, 0)       # frame 0 for the frames whose window does not reach it
    temporal = _band(c["fh"], c["fh"] // 4) * _band(c["fw"], c["fw"] // 4) if c["window_2d"] else _band(S, ws)
    kept = sum(1 for y in range(c["fh"]) for x in range(c["fw"]) if y % 2 == x % 2)
    per = {"frame": spatial * S * S + text, "position": temporal * T * T + text, "lowrank": N * (T * kept + L)}
    if c["amp"] < 1:                        # the planted structure is too weak for Algorithm 1: every head is Textural
        per["frame"] = per["position"] = per["lowrank"]
    return c["B"] * sum(per[k] for k in _kinds(c))


def work(case):
    c = case
    Nv, S, heads = c["T"] * c["fh"] * c["fw"], c["fh"] * c["fw"], c["B"] * c["H"]
    rows = heads * (Nv + c["L"])
    flops = 4.0 * c["D"] * _pairs(c)
    if c["kind"] != "dense":                # ARM: Q K^T of the sampled tokens
        n = math.ceil(Nv / c["omega"])
        flops += 2.0 * c["D"] * heads * (n * n + (S * S if c["mode"] == 0 else 0))
    return {"bytes": 4 * rows * c["D"] * 2 + (rows * 4 if c["lse"] else 0), "flops": flops}


def tolerance(case):
    # bf16 outputs of bf16-rounded weights.  Against the same attention in 64 bits a dense call is off by rel 1.6e-3 to
    # 2.2e-3 and max 5e-3 to 1.44e-2 (heads of the tiny, ragged, 8x1024 and CogVideoX shapes): four times that.  Head
    # classes and windows are exact: the planted structure leaves no recall near the threshold.
    return {"rel": 7e-3, "max": 6e-2}


def _kept(c, kind, window, rows, cols):
    """Which of the pairs (row token, key token) a head of this kind keeps, by the definitions of the patterns; `rows`
    and `cols` are token indices in original order."""
    S, W, Nv = c["fh"] * c["fw"], c["fw"], c["T"] * c["fh"] * c["fw"]
    if kind == TEXTURAL:
        p = cols % S
        return ((cols >= Nv) | ((p // W) % 2 == (p % W) % 2)).expand(len(rows), -1)
    r, u = rows[:, None], cols[None, :]
    if kind == SPATIAL:
        keep = (r // S - u // S).abs() <= window
        if c["key_frame"]:
            keep |= u < S
    elif c["window_2d"]:
        pr, pu = r % S, u % S
        keep = ((pr // W - pu // W).abs() <= c["fh"] // 4) & ((pr % W - pu % W).abs() <= c["fw"] // 4)
    else:
        keep = (r % S - u % S).abs() <= window
    return keep | (r >= Nv) | (u >= Nv)


def _recalls(c, q, k, tokens, kind, windows):
    """Mean share of the softmax mass that each window of a pattern keeps among the sampled tokens (64 bits)."""
    got = torch.zeros(len(windows), dtype=torch.float64, device=q.device)
    scaled, keys = q[tokens].double() / math.sqrt(c["D"]), k[tokens].double()
    for r0 in range(0, len(tokens), 4096):
        p = torch.softmax(scaled[r0:r0 + 4096] @ keys.T, dim=-1)
        for i, w in enumerate(windows):
            got[i] += (p * _kept(c, kind, w, tokens[r0:r0 + 4096], tokens)).sum()
    return (got / len(tokens)).tolist()


def _classify(c, q, k):
    """(class, window) of one head by Algorithm 1, or by the smallest bandwidth that qualifies."""
    T, S = c["T"], c["fh"] * c["fw"]
    every = torch.arange(0, T * S, c["omega"], device=q.device)
    first = torch.arange(S, device=q.device) if c["mode"] == 0 else every
    wf, ws = _windows(c)
    plus = c["kind"] == "plus"
    wt = [int(b * S) for b in BANDWIDTHS] if plus else [ws]
    wsp = [int(b * T) for b in BANDWIDTHS] if plus else [wf]
    for kind, tokens, windows in ((TEMPORAL, first, wt), (SPATIAL, every, wsp)):
        for w, recall in zip(windows, _recalls(c, q, k, tokens, kind, windows)):
            if recall >= 0.9:
                return kind, w
    return TEXTURAL, -1


def exact(case, seed):
    """`run`'s outputs from the definitions in 64 bits: explicit masks, explicit softmax, a block of rows at a time."""
    c = case
    q, k, v = _inputs(c, seed)
    B, H, N, D = q.shape
    if B * H * float(N) * N * D > MOST_EXACT:
        return None
    dev = q.device
    tokens = torch.arange(N, device=dev)
    o = torch.empty(q.shape, dtype=torch.float64, device=dev)
    lse = torch.empty(q.shape[:3], dtype=torch.float64, device=dev)
    classes, windows = (torch.full((B, H), -1, dtype=torch.int32, device=dev) for _ in range(2))
    for b in range(B):
        for h in range(H):
            keep_all, cols = c["kind"] == "dense", tokens
            if not keep_all:
                kind, window = _classify(c, q[b, h], k[b, h])
                classes[b, h], windows[b, h] = kind, window
                if kind == TEXTURAL:
                    cols, keep_all = tokens[_kept(c, kind, 0, tokens[:1], tokens)[0]], True
            keys, values = k[b, h][cols].double(), v[b, h][cols].double()
            step = max(128, (1 << 28) // len(cols))
            for r0 in range(0, N, step):
                rows = tokens[r0:r0 + step]
                s = (q[b, h][rows].double() / math.sqrt(D)) @ keys.T
                if not keep_all:
                    s.masked_fill_(~_kept(c, kind, window, rows, cols), -math.inf)
                top = s.amax(dim=1, keepdim=True)
                s.sub_(top).exp_()
                total = s.sum(dim=1, keepdim=True)
                o[b, h, r0:r0 + step] = (s @ values).div_(total)
                lse[b, h, r0:r0 + step] = (top + total.log())[:, 0]
    if c["kind"] == "host":
        return {"o": o}
    out = {"o": o, "lse": lse if c["lse"] else None}
    if c["kind"] != "dense":
        out["head_class"] = classes
    if c["kind"] == "plus":
        out["head_window"] = windows
    return out
